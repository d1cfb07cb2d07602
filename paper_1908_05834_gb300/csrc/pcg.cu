// Preconditioned conjugate gradients on the normal equations of the
// minimisation: one kernel for both solves of an interior-point iteration, with
// the iteration's passes over the entries around them (ip.cuh).
//
// Each iteration is a product with the finest level, a vector update and one
// V-cycle (a damped-Jacobi sweep before and after the coarse correction, the
// coarsest level solved by its inverse): two dependent passes per level and
// three more.  Launched pass by pass they cost 2.5 us each whatever their size,
// plus one block cycling every level of up to 4 096 nodes through global memory
// with 40 sweeps at the bottom: 0.13 ms per iteration at 32^2, 0.22 ms at
// 128^2, 0.35 ms at 24^3, for 5 to 30 us of arithmetic and memory traffic.
//
// In one launch what bounds a solve is, per pass, the barrier after
// it (2 350 clocks across the grid, about 450 within a cluster), one round trip
// to L2 (~800 clocks), and the FP64 pipe: a warp instruction of it takes 19
// clocks of its SM however many lanes are active, so work is spread over many
// SMs even when there is little of it, sums take one thread per row, and scalars
// are computed by one thread.  So:
//   - restriction is fused with the residual and the next level's first sweep,
//     prolongation with the sweep of the level above: one pass down and one up;
//   - a block owns the rows of its aggregates' members for the whole solve and
//     keeps them (columns, weights, diagonals, vectors) in shared memory as far
//     as they fit, finest level first.  A pass first gathers the vector for all of
//     its entries at once (one round trip), then sums rows from shared memory;
//   - the levels of at most kTierEntries entries are cycled by the first cluster,
//     rows and vectors spread over its blocks' shared memory (a pass gathers
//     through distributed shared memory, cluster barriers between the passes);
//     those of at most kCopyNodes nodes are held and cycled whole by every block
//     of it, with block barriers alone;
//   - a system of at most kSmallNodes nodes is solved by one cluster of
//     kSmallCluster blocks alone, the finest level like the others;
//   - the stopping test runs on the device, identically in every block.
// Levels too large for shared memory take a general path that reads rows and
// vectors from global memory, several lanes per row.
#include "amg.cuh"
#include "device.cuh"
#include "gridbar.cuh"
#include "ip.cuh"

namespace bchar {

constexpr int kNT = kSolveThreads;
// Levels of at most this many entries (and nodes) belong to the first cluster:
// at 16 000 entries a pass of 8 blocks costs about what the grid's barrier does.
constexpr int64_t kTierEntries = 16000;
constexpr int kTierNodes = 3000;
// Levels of at most this many nodes (and entries) are cycled by every block of
// the cluster for itself: 4 warps of rows, about 1 500 clocks a pass, where the
// exchange through the cluster takes 1 000 beyond the arithmetic.
constexpr int kCopyNodes = 64;
constexpr int64_t kCopyEntries = 2000;
// entries per block beyond which the general path forms p in a pass of its own
// instead of twice the gathers and products per entry
constexpr int64_t kFuseEntries = 5000;

struct PcgArgs {
    HierView v;
    int n0;
    int64_t e0;
    int schur;
    int64_t nc;
    const int64_t *row_ptr, *col_ptr;
    const int32_t *col, *csc_row;
    const double *a2, *a2c, *diag, *rhs;      // the system on rows and columns
    double *dy;                               // its solution
    double *d, *r, *p0, *p1, *q, *z, *ib;     // finest level; ib: 1 / target of each constraint
    const double *b_row, *volphi;
    IpArgs ip;
    SolveTols tols;   // predictor (from zero), corrector (from the predictor's d)
    int vcycle;       // 1: one V-cycle only (timing)
    unsigned smem;    // dynamic shared memory
};

// ---------------------------------------------------------------- clusters

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Address of this shared-memory place in block r of the cluster.
__device__ __forceinline__ unsigned remote(const void *p, unsigned r) {
    const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(r));
    return ra;
}
__device__ __forceinline__ double load_remote(unsigned a) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void store_remote(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// Stores v at this shared-memory place of every block of the cluster.
__device__ __forceinline__ void store_all(double *p, double v, unsigned nr) {
    for (unsigned r = 0; r < nr; ++r) store_remote(remote(p, r), v);
}

// ---------------------------------------------------------------- shares of a level

// The rows of one block: the members of its aggregates in aggregate order, then
// nodes without a coarse counterpart; on a coarsest level a range of nodes.
struct Rows {
    int64_t noff;       // the level's first node
    int n, nrow, nmem;  // level nodes; rows here, of which in aggregates
    int ngrp, i0;       // aggregates here, the first one
    int ents;
    int here;           // 1: all of it in shared memory, 2: without room for a pass's gathered values
    int lpr, lprg;      // general path: lanes per row, per aggregate
    int lg;             // log2 of the lanes per row with the rows in shared memory
    int m0, l0;         // general path: where the rows are in the level's order array
    int whole;          // a coarsest level: rows i0 ..
    // places in shared memory (byte offsets): row's node, entries; aggregate's rows; row's members in the finer
    // level; the rows by length
    unsigned id, off, col, gst, mst, mem, ord;
    unsigned w, dg, om, omc, res, bo, mx;
    // the first cluster's levels: the vector (spread: this block's range of nodes; else all of it).
    // Spread levels hold addresses in the cluster's shared memory: of the row's own value (xa), its entries'
    // values (col) and, when the finer level is spread too, its members' (mem).
    int kind;
    unsigned x, xa, db;
};

extern __shared__ __align__(16) unsigned char g_smem[];

__device__ __forceinline__ double *at_d(unsigned o) { return reinterpret_cast<double *>(g_smem + o); }
__device__ __forceinline__ int *at_i(unsigned o) { return reinterpret_cast<int *>(g_smem + o); }

// The same with pointers, in registers for the length of a pass: loading each
// pointer where it is used would put two shared-memory latencies on every access.
struct View {
    int n, nrow, nmem, ngrp, i0, ents, lg;
    unsigned db;  // spread and copied levels: from a value of x to that of b
    int *id, *off, *col, *gst, *mst, *mem, *ord;
    double *w, *dg, *om, *omc, *res, *bo, *mx, *x;
    unsigned *xa;
};
__device__ __forceinline__ View view(const Rows &R) {
    View v;
    v.n = R.n;
    v.nrow = R.nrow;
    v.nmem = R.nmem;
    v.ngrp = R.ngrp;
    v.i0 = R.i0;
    v.ents = R.ents;
    v.lg = R.lg;
    v.db = R.db;
    v.id = at_i(R.id);
    v.off = at_i(R.off);
    v.col = at_i(R.col);
    v.gst = at_i(R.gst);
    v.mst = at_i(R.mst);
    v.mem = at_i(R.mem);
    v.ord = at_i(R.ord);
    v.w = at_d(R.w);
    v.dg = at_d(R.dg);
    v.om = at_d(R.om);
    v.omc = at_d(R.omc);
    v.res = at_d(R.res);
    v.bo = at_d(R.bo);
    v.mx = at_d(R.mx);
    v.x = at_d(R.x);
    v.xa = reinterpret_cast<unsigned *>(at_i(R.xa));
    return v;
}
enum { kGrid = 0, kSpread = 1, kCopy = 2 };

struct Shared {
    Rows lev[kMaxLevels];
    double sum[2][16];
    unsigned long long max[16];
    double out[3];
    double alpha, beta, rz, inv_rz, res_max;
    int conv;
    int tmp[33];
    int nlev, t0, tr, dense, sweeps;  // t0: first level of the first cluster, tr: first copied one
    // places in shared memory: second vector of a coarsest level; the coarsest level's inverse; gathered values of a pass (spread levels, grid levels); small systems: z and two directions
    // (spread like x of the finest level), the blocks' parts of the dot products; finest level, own rows
    unsigned alt, inv, xs, xg, zv, pv, dots, ro, dd, qo, po, zo, ibo;
};

// Claims room for n values at p (an offset in the dynamic shared memory).
template <class T> __device__ __forceinline__ unsigned take_n(unsigned &p, int n) {
    const unsigned q = p;
    p += (static_cast<unsigned>(sizeof(T)) * static_cast<unsigned>(n > 0 ? n : 1) + 15u) & ~15u;
    return q;
}

__device__ __forceinline__ int scan_nt(int x, int *tmp, int &total) {  // exclusive, over kNT threads
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = x;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();
    if (lane == 31) tmp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int t = lane < kNT / 32 ? tmp[lane] : 0;
        int s = t;
        for (int o = 1; o < 32; o <<= 1) {
            const int q = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += q;
        }
        tmp[lane] = s - t;
        if (lane == 31) tmp[32] = s;
    }
    __syncthreads();
    total = tmp[32];
    return tmp[wid] + incl - x;
}

// Lanes per item of the general path: enough to keep the block's threads busy,
// but at least two entries each.
__device__ __forceinline__ int lanes_for_items(int items, double mean) {
    int l = 1;
    while (l < 16 && 4 * l <= mean && items * 2 * l <= kNT) l *= 2;
    return l;
}

__device__ __forceinline__ void chunk(int n, int r, int nr, int &c0, int &c1) {
    const int ch = (n + nr - 1) / nr;
    c0 = min(n, r * ch);
    c1 = min(n, c0 + ch);
}

// Loads a share of level l: rank r's (of nr) part of a spread level, all of a
// copied one, or the block's Seg of the build of a grid level.  A grid level's
// share is kept only when it fits with keep bytes to spare and room for a pass's
// gathered values (most: those of the levels loaded before).  False: it does not
// fit.  Block-collective.
__device__ bool load_rows(const HierView &v, Shared &sh, int l, int kind, int r, int nr, unsigned &p, unsigned end,
                          size_t keep, int most) {
    const LevelInfo L = v.H->L[l];
    const bool coarsest = l == sh.nlev - 1, grid = kind == kGrid;
    Rows &R = sh.lev[l];
    const int64_t noff = L.noff, noff2 = noff + L.n;
    const int nco = coarsest ? 0 : v.H->L[l + 1].n;
    int I0 = 0, I1 = 0, l0 = 0, lv = 0, m0 = 0;
    if (!grid && kind == kCopy) {
        r = 0;
        nr = 1;
    }
    if (coarsest) {
        chunk(L.n, r, nr, I0, I1);
    } else if (!grid) {
        int a, b;
        chunk(nco, r, nr, I0, I1);
        chunk(L.n - L.nmem, r, nr, a, b);
        l0 = L.nmem + a;
        lv = b - a;
    } else {
        const Seg g = L.grid || r == 0 ? v.seg[l * kMaxCtas + r] : Seg{};  // a level built by block 0 is block 0's
        I0 = g.g0;
        I1 = g.g0 + g.glen;
        l0 = g.l0;
        lv = g.llen;
        m0 = g.m0;
    }
    const int tid = threadIdx.x;
    int mine = 0, nmem = 0;
    if (!coarsest)
        for (int I = I0 + tid; I < I1; I += kNT) mine += v.gc[noff2 + I];
    scan_nt(mine, sh.tmp, nmem);
    const int ngrp = coarsest ? 0 : I1 - I0, nrow = coarsest ? I1 - I0 : nmem + lv;
    __syncthreads();
    if (tid == 0) {
        R.noff = noff;
        R.n = L.n;
        R.nrow = nrow;
        R.nmem = nmem;
        R.ngrp = ngrp;
        R.i0 = I0;
        R.here = 0;
        R.kind = kind;
        R.m0 = m0;
        R.l0 = l0;
        R.whole = coarsest ? 1 : 0;
        const double mean = static_cast<double>(L.nnz) / (L.n > 0 ? L.n : 1);
        R.lpr = lanes_for_items((L.n + nr - 1) / nr, mean);
        R.lprg = lanes_for_items((nco + nr - 1) / nr, mean * L.n / (nco > 0 ? nco : 1));
    }
    const size_t node_bytes = static_cast<size_t>(nrow) * (4 * 5 + 8 * 4) + static_cast<size_t>(ngrp) * 12 + 16 * 16;
    __syncthreads();
    if (static_cast<size_t>(end - p) < node_bytes + keep) return false;  // block-uniform
    const unsigned p_before = p;
    Rows N = R;
    N.id = take_n<int>(p, nrow);
    N.off = take_n<int>(p, nrow + 1);
    N.gst = take_n<int>(p, ngrp + 1);
    N.mst = take_n<int>(p, nrow + 1);
    N.xa = take_n<unsigned>(p, kind == kSpread ? nrow : 1);
    N.ord = take_n<int>(p, nrow);
    N.dg = take_n<double>(p, nrow);
    N.om = take_n<double>(p, nrow);
    N.omc = take_n<double>(p, ngrp);
    N.res = take_n<double>(p, nrow);
    N.bo = take_n<double>(p, nrow);
    int *const id = at_i(N.id), *const off = at_i(N.off), *const gst = at_i(N.gst), *const mst = at_i(N.mst);
    unsigned *const xa = reinterpret_cast<unsigned *>(at_i(N.xa));
    double *const dg = at_d(N.dg), *const om = at_d(N.om), *const omc = at_d(N.omc);
    const double *const x = at_d(R.x);
    // rows
    int run = 0;
    for (int base = 0; base < ngrp; base += kNT) {
        const int g = base + tid;
        const int c = g < ngrp ? v.gc[noff2 + I0 + g] : 0;
        int tot;
        const int at = run + scan_nt(c, sh.tmp, tot);
        if (g < ngrp) {
            gst[g] = at;
            omc[g] = v.om[noff2 + I0 + g];
            const int64_t o = noff + v.gs[noff2 + I0 + g];
            for (int q = 0; q < c; ++q) id[at + q] = v.own[o + q];
        }
        run += tot;
    }
    if (tid == 0) gst[ngrp] = run;
    if (coarsest)
        for (int k = tid; k < nrow; k += kNT) id[k] = I0 + k;
    else
        for (int k = tid; k < lv; k += kNT) id[nmem + k] = v.own[noff + l0 + k];
    __syncthreads();
    const int cx = (L.n + nr - 1) / nr;  // nodes per block of a spread vector
    int ents = 0, mems = 0;
    for (int base = 0; base < nrow; base += kNT) {
        const int k = base + tid;
        const int i = k < nrow ? id[k] : 0;
        const int len = k < nrow ? v.rl[noff + i] : 0;
        const int gm = k < nrow && l > 0 ? v.gc[noff + i] : 0;
        int tot;
        const int at = scan_nt(len, sh.tmp, tot);
        int mtot;
        const int mat = scan_nt(gm, sh.tmp, mtot);
        if (k < nrow) {
            off[k] = ents + at;
            mst[k] = mems + mat;
            dg[k] = v.dg[noff + i];
            om[k] = v.om[noff + i];
            if (kind == kSpread) xa[k] = remote(x + i % cx, i / cx);
        }
        ents += tot;
        mems += mtot;
    }
    if (tid == 0) {
        off[nrow] = ents;
        mst[nrow] = mems;
    }
    __syncthreads();
    const size_t need = static_cast<size_t>(mems) * (kind == kCopy ? 4 : 12) + static_cast<size_t>(ents) * 12 + 6 * 16;
    const size_t stage = kind == kCopy ? 0 : static_cast<size_t>(max(ents, most)) * 8 + 32;
    const bool staged = static_cast<size_t>(end - p) >= need + keep + stage;
    if (!staged && (!grid || static_cast<size_t>(end - p) < need + keep + static_cast<size_t>(most) * 8 + 32)) {
        p = p_before;
        return false;
    }
    // A warp's FP64 time is its longest row's, so threads take the rows by length
    // (ranks by counting: ties in row order, the sums stay reproducible).
    int *const ord = at_i(N.ord);
    for (int k = tid; k < nrow; k += kNT) {
        const int len = off[k + 1] - off[k];
        int at = k;
        if (nrow <= kNT) {
            at = 0;
            for (int q = 0; q < nrow; ++q) {
                const int o = off[q + 1] - off[q];
                at += o > len || (o == len && q < k) ? 1 : 0;
            }
        }
        ord[at] = k;
    }
    N.mem = take_n<int>(p, mems);
    N.mx = kind == kCopy ? 0 : take_n<double>(p, mems);
    int *const mem = at_i(N.mem);
    if (l > 0) {
        const LevelInfo F = v.H->L[l - 1];
        const bool addr = kind == kSpread && sh.lev[l - 1].kind == kSpread && l - 1 >= sh.t0;
        const int cf = (F.n + nr - 1) / nr;
        for (int k = tid; k < nrow; k += kNT) {
            const int64_t o = F.noff + v.gs[noff + id[k]];
            for (int q = mst[k]; q < mst[k + 1]; ++q) {
                const int i = v.own[o + q - mst[k]];
                mem[q] = addr ? static_cast<int>(remote(at_d(sh.lev[l - 1].x) + i % cf, i / cf)) : i;
            }
        }
    }
    N.w = take_n<double>(p, ents);
    N.col = take_n<int>(p, ents);
    N.ents = ents;
    // up to four warps of rows: more lanes per row than that and the FP64 pipe's slots cost more
    // than the shorter sums save
    N.lg = 0;
    while (N.lg < 3 && (nrow << (N.lg + 1)) <= 128) ++N.lg;
    N.here = staged ? 1 : 2;
    double *const w = at_d(N.w);
    int *const col = at_i(N.col);
    const int lane = tid & 31;
    for (int k = tid >> 5; k < nrow; k += kNT / 32) {
        const int64_t e = v.rs[noff + id[k]];
        for (int q = lane; q < off[k + 1] - off[k]; q += 32) {
            const int c = v.ecol[e + q];
            col[off[k] + q] = kind == kSpread ? static_cast<int>(remote(x + c % cx, c / cx)) : c;
            w[off[k] + q] = v.ew[e + q];
        }
    }
    __syncthreads();
    if (tid == 0) R = N;
    __syncthreads();
    return true;
}

// ---------------------------------------------------------------- sums over blocks

// Non-negative doubles compare like their bits as integers, without the FP64 pipe.
__device__ __forceinline__ unsigned long long bits_of(double v) {
    return static_cast<unsigned long long>(__double_as_longlong(v));
}
__device__ __forceinline__ unsigned long long max_bits(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

// The threads' parts of two sums and the bits of a maximum (of the first
// `active` threads; the others have none) into sh.out, where thread s < slots
// may read its own; fixed order.
__device__ __forceinline__ void block_partials(Shared &sh, int slots, int active, double a, double b,
                                               unsigned long long mx) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nw = min(kNT / 32, (active + 31) >> 5);
    if (wid < nw) {  // warp-uniform
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            if (slots > 1) {
                b += __shfl_xor_sync(0xffffffffu, b, o);
                mx = max_bits(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            }
        }
        if (lane == 0) {
            sh.sum[0][wid] = a;
            sh.sum[1][wid] = b;
            sh.max[wid] = mx;
        }
    }
    __syncthreads();
    if (tid < slots) {
        if (tid == 2) {
            unsigned long long m = 0;
            for (int q = 0; q < nw; ++q) m = max_bits(m, sh.max[q]);
            sh.out[2] = __longlong_as_double(static_cast<long long>(m));
        } else {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            for (int q = 0; q < nw; q += 4) {
                s0 += sh.sum[tid][q];
                if (q + 1 < nw) s1 += sh.sum[tid][q + 1];
                if (q + 2 < nw) s2 += sh.sum[tid][q + 2];
                if (q + 3 < nw) s3 += sh.sum[tid][q + 3];
            }
            sh.out[tid] = (s0 + s1) + (s2 + s3);
        }
    }
    __syncwarp();
}

// The totals of the blocks' partials part[slot][0 .. nb) (slot < slots, stride
// apart) into sh.out, one warp per slot; the block is synchronised after it.
__device__ __forceinline__ void block_totals(Shared &sh, const double *part, int stride, int slots, unsigned nb) {
    const int lane = threadIdx.x & 31, s = threadIdx.x >> 5;
    if (s < slots) {
        double x[kMaxCtas / 32];
#pragma unroll
        for (int k = 0; k < kMaxCtas / 32; ++k) {
            const unsigned q = k * 32 + lane;
            x[k] = q < nb ? *reinterpret_cast<const volatile double *>(part + s * stride + q) : 0.0;
        }
        double y;
        if (s == 2) {
            unsigned long long m = 0;
#pragma unroll
            for (int k = 0; k < kMaxCtas / 32; ++k) m = max_bits(m, bits_of(x[k]));
            for (int o = 16; o > 0; o >>= 1) m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
            y = __longlong_as_double(static_cast<long long>(m));
        } else {
            double u = x[0], t = nb > 32 ? x[1] : 0.0;
#pragma unroll
            for (int k = 2; k < kMaxCtas / 32; k += 2)
                if (k * 32 < static_cast<int>(nb)) {
                    u += x[k];
                    t += x[k + 1];
                }
            y = nb > 32 ? u + t : u;
            for (int o = nb > 16 ? 16 : 8; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        }
        if (lane == 0) sh.out[s] = y;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- general path (vectors, and rows unless they fit, from global memory)

struct Row {
    int id, len;
    const int *col;
    const double *w;
    double dg, om;
};

// HERE: from shared memory.  As a template parameter of the passes: with a pointer
// that may be to either memory (generic loads) a system whose rows fit but for the
// gathered values took 325 ms a step instead of 277 (32^3, rows of 5 to 40).
template <bool HERE> __device__ __forceinline__ Row row_at(const HierView &v, const Rows &R, int k) {
    Row r;
    if (HERE) {
        const int o = at_i(R.off)[k];
        r.id = at_i(R.id)[k];
        r.len = at_i(R.off)[k + 1] - o;
        r.col = at_i(R.col) + o;
        r.w = at_d(R.w) + o;
        r.dg = at_d(R.dg)[k];
        r.om = at_d(R.om)[k];
        return r;
    }
    r.id = R.whole ? R.i0 + k : v.own[R.noff + (k < R.nmem ? R.m0 + k : R.l0 + k - R.nmem)];
    const int64_t e = v.rs[R.noff + r.id];
    r.len = v.rl[R.noff + r.id];
    r.col = v.ecol + e;
    r.w = v.ew + e;
    r.dg = v.dg[R.noff + r.id];
    r.om = v.om[R.noff + r.id];
    return r;
}

__device__ __forceinline__ int row_id(const HierView &v, const Rows &R, int k) {
    if (R.here) return at_i(R.id)[k];
    return R.whole ? R.i0 + k : v.own[R.noff + (k < R.nmem ? R.m0 + k : R.l0 + k - R.nmem)];
}

template <int LPR> __device__ __forceinline__ double lanes_sum(double s) {
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// sum of w_j x_j over this lane's entries of a row
template <int LPR> __device__ __forceinline__ double lane_dot(const Row &r, int sub, const double *x) {
    double s = 0.0;
    int e = sub;
    for (; e + 3 * LPR < r.len; e += 4 * LPR) {
        const double x0 = x[r.col[e]], x1 = x[r.col[e + LPR]], x2 = x[r.col[e + 2 * LPR]], x3 = x[r.col[e + 3 * LPR]];
        s += r.w[e] * x0;
        s += r.w[e + LPR] * x1;
        s += r.w[e + 2 * LPR] * x2;
        s += r.w[e + 3 * LPR] * x3;
    }
    for (; e < r.len; e += LPR) s += r.w[e] * x[r.col[e]];
    return s;
}

// Runs f(ok, sub, k) over items k < n, LPR lanes each; every lane of a warp
// runs the same number of rounds, so f may shuffle.
template <int LPR, class F> __device__ __forceinline__ void for_items(int n, F f) {
    const int lane = threadIdx.x & 31;
    for (int k0 = static_cast<int>(threadIdx.x >> 5) * (32 / LPR); k0 < n; k0 += kNT / LPR) {
        const int k = k0 + lane / LPR;
        f(k < n, lane % LPR, k);
    }
}

// Lanes per row of the general passes: with many rows per block, else they are in
// shared memory.  A single cluster's system comes here only when its levels do not
// fit: one variant is enough.
#define WITH_LANES(L, H, CALL)                                  \
    if constexpr (Bar::kCluster) {                              \
        constexpr bool HERE = false;                            \
        constexpr int LPR = 4;                                  \
        CALL;                                                   \
    } else if (H) {                                             \
        constexpr bool HERE = true;                             \
        WITH_LANES_OF(L, CALL)                                  \
    } else {                                                    \
        constexpr bool HERE = false;                            \
        WITH_LANES_OF(L, CALL)                                  \
    }
#define WITH_LANES_OF(L, CALL)                                  \
    switch (L) {                                                \
    case 1: { constexpr int LPR = 1; CALL; } break;             \
    case 2: { constexpr int LPR = 2; CALL; } break;             \
    case 4: { constexpr int LPR = 4; CALL; } break;             \
    case 8: { constexpr int LPR = 8; CALL; } break;             \
    default: { constexpr int LPR = 16; CALL; } break;           \
    }

// b and x of the next level: the residual b - L x summed over each aggregate,
// and that level's first sweep from zero.
template <int LPR, bool HERE>
__device__ void general_down(const HierView &v, const Rows &R, const double *bl, const double *x, double *bc, double *xc) {
    const int64_t noff2 = R.noff + R.n;
    for_items<LPR>(R.ngrp, [&](bool ok, int sub, int g) {
        double s = 0.0;
        if (ok) {
            const int k0 = HERE ? at_i(R.gst)[g] : v.gs[noff2 + R.i0 + g] - R.m0;
            const int k1 = HERE ? at_i(R.gst)[g + 1] : k0 + v.gc[noff2 + R.i0 + g];
            for (int k = k0; k < k1; ++k) {
                const Row r = row_at<HERE>(v, R, k);
                if (sub == 0) s += bl[r.id] - r.dg * x[r.id];
                s += lane_dot<LPR>(r, sub, x);
            }
        }
        s = lanes_sum<LPR>(s);
        if (ok && sub == 0) {
            bc[R.i0 + g] = s;
            xc[R.i0 + g] = v.om[noff2 + R.i0 + g] * s;
        }
    });
}

// Adds val to x of node i's members in the finer level (a node's lanes share them).
__device__ __forceinline__ void prolong(const HierView &v, int64_t noff, int64_t fine, int i, double val, int sub, int lpr,
                                        double *xf) {
    const int g = v.gs[noff + i], c = v.gc[noff + i];
    for (int k = sub; k < c; k += lpr) xf[v.own[fine + g + k]] += val;
}

// The sweep after the coarse correction, prolonged into the finer level.
template <int LPR, bool HERE>
__device__ void general_up(const HierView &v, const Rows &R, const double *bl, const double *x, int64_t fine, double *xf) {
    for_items<LPR>(R.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        double xi = 0.0, bi = 0.0;
        if (ok) {
            r = row_at<HERE>(v, R, k);
            xi = x[r.id];
            bi = bl[r.id];
            s = lane_dot<LPR>(r, sub, x);
        }
        s = lanes_sum<LPR>(s);
        if (ok) prolong(v, R.noff, fine, r.id, xi + r.om * (bi - (r.dg * xi - s)), sub, LPR, xf);
    });
}

// The same on the finest level: z, and this thread's parts of z.r and z.q.
template <int LPR, bool HERE>
__device__ void general_top(const HierView &v, const Rows &R, const double *r_, const double *q_, const double *x, double *z,
                            double &rz, double &zq) {
    for_items<LPR>(R.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        double xi = 0.0, bi = 0.0, qi = 0.0;
        if (ok) {
            r = row_at<HERE>(v, R, k);
            xi = x[r.id];
            bi = r_[r.id];
            qi = q_[r.id];
            s = lane_dot<LPR>(r, sub, x);
        }
        s = lanes_sum<LPR>(s);
        if (ok && sub == 0) {
            const double zi = xi + r.om * (bi - (r.dg * xi - s));
            z[r.id] = zi;
            rz += zi * bi;
            zq += zi * qi;
        }
    });
}

// One Jacobi sweep of a coarsest level shared by all blocks.
template <int LPR, bool HERE>
__device__ void general_sweep(const HierView &v, const Rows &R, const double *bl, const double *x, double *xo) {
    for_items<LPR>(R.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        if (ok) {
            r = row_at<HERE>(v, R, k);
            s = lane_dot<LPR>(r, sub, x);
        }
        s = lanes_sum<LPR>(s);
        if (ok && sub == 0) {
            const double xi = x[r.id];
            xo[r.id] = xi + r.om * (bl[r.id] - (r.dg * xi - s));
        }
    });
}

// q = L p and this thread's part of p.q.  FUSED: p = z + beta pold is formed by
// its readers and stored by its owner.
template <int LPR, bool HERE, bool FUSED>
__device__ void general_product(const HierView &v, const Rows &R, const double *z, const double *pold, double beta,
                                double *p, double *q, double &pq) {
    for_items<LPR>(R.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0, pi = 0.0;
        Row r{};
        if (ok) {
            r = row_at<HERE>(v, R, k);
            if (FUSED) {
                pi = z[r.id] + beta * pold[r.id];
                int e = sub;
                for (; e + LPR < r.len; e += 2 * LPR) {
                    const int c0 = r.col[e], c1 = r.col[e + LPR];
                    const double z0 = z[c0], o0 = pold[c0], z1 = z[c1], o1 = pold[c1];
                    s += r.w[e] * (z0 + beta * o0);
                    s += r.w[e + LPR] * (z1 + beta * o1);
                }
                if (e < r.len) {
                    const int c0 = r.col[e];
                    s += r.w[e] * (z[c0] + beta * pold[c0]);
                }
            } else {
                pi = p[r.id];
                s = lane_dot<LPR>(r, sub, p);
            }
        }
        s = lanes_sum<LPR>(s);
        if (ok && sub == 0) {
            const double qi = r.dg * pi - s;
            if (FUSED) p[r.id] = pi;
            q[r.id] = qi;
            pq += pi * qi;
        }
    });
}

// ---------------------------------------------------------------- shared levels with the rows in shared memory

// Runs f(ok, sub, t) over t < n with 2^lg lanes each; every lane of a warp runs
// the same number of rounds, so f may shuffle.
template <class F> __device__ __forceinline__ void for_rows(int n, int lg, F f) {
    const int tid = threadIdx.x;
    for (int t0 = (tid & ~31) >> lg; t0 < n; t0 += kNT >> lg) {
        const int t = t0 + ((tid & 31) >> lg);
        f(t < n, tid & ((1 << lg) - 1), t);
    }
}

__device__ __forceinline__ double lanes_total(double s, int lg) {
    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// s plus this lane's part of sum w_e x_e over row k's entries, xs[e] the gathered
// values; independent chains (a dependent FP64 product takes 65 clocks, its issue
// slot 19)
__device__ __forceinline__ double row_sum(const View &R, int k, int sub, const double *xs, double s) {
    const int step = 1 << R.lg, e1 = R.off[k + 1];
    int e = R.off[k] + sub;
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (; e + 3 * step < e1; e += 4 * step) {
        s += R.w[e] * xs[e];
        s1 += R.w[e + step] * xs[e + step];
        s2 += R.w[e + 2 * step] * xs[e + 2 * step];
        s3 += R.w[e + 3 * step] * xs[e + 3 * step];
    }
    if (e + step < e1) {
        s += R.w[e] * xs[e];
        s1 += R.w[e + step] * xs[e + step];
        e += 2 * step;
    }
    if (e < e1) s2 += R.w[e] * xs[e];
    return (s + s1) + (s2 + s3);
}

// the same over a copied level, from the vector itself
__device__ __forceinline__ double copy_sum(const View &R, int k, int sub, const double *x, double s) {
    const int step = 1 << R.lg, e1 = R.off[k + 1];
    int e = R.off[k] + sub;
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (; e + 3 * step < e1; e += 4 * step) {
        const double x0 = x[R.col[e]], x1 = x[R.col[e + step]], x2 = x[R.col[e + 2 * step]], x3 = x[R.col[e + 3 * step]];
        s += R.w[e] * x0;
        s1 += R.w[e + step] * x1;
        s2 += R.w[e + 2 * step] * x2;
        s3 += R.w[e + 3 * step] * x3;
    }
    if (e + step < e1) {
        s += R.w[e] * x[R.col[e]];
        s1 += R.w[e + step] * x[R.col[e + step]];
        e += 2 * step;
    }
    if (e < e1) s2 += R.w[e] * x[R.col[e]];
    return (s + s1) + (s2 + s3);
}

// sum of the residuals of aggregate g's rows
__device__ __forceinline__ double group_sum(const View &R, int g) {
    int k = R.gst[g];
    const int k1 = R.gst[g + 1];
    double s0 = R.res[k], s1 = k + 1 < k1 ? R.res[k + 1] : 0.0;
    for (k += 2; k < k1; k += 2) {
        s0 += R.res[k];
        if (k + 1 < k1) s1 += R.res[k + 1];
    }
    return s0 + s1;
}

__device__ void fast_down(const Shared &sh, const View R, const double *bl, const double *x, double *bc, double *xc) {
    const int tid = threadIdx.x;
    double *const xg = at_d(sh.xg);
    const double *const ro = at_d(sh.ro);
    for (int e = tid; e < R.ents; e += kNT) xg[e] = x[R.col[e]];
    for (int k = tid; k < R.nrow; k += kNT) {
        const int i = R.id[k];
        const double xi = x[i], bi = bl ? bl[i] : ro[k];
        R.bo[k] = bi;
        R.res[k] = xi;
    }
    __syncthreads();
    for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
        const int k = ok ? R.ord[t] : 0;
        const bool in = ok && k < R.nmem;
        double s = 0.0;
        if (in) s = row_sum(R, k, sub, xg, sub ? 0.0 : R.bo[k] - R.dg[k] * R.res[k]);
        s = lanes_total(s, R.lg);
        if (in && sub == 0) R.res[k] = s;
    });
    __syncthreads();
    for (int g = tid; g < R.ngrp; g += kNT) {
        const double s = group_sum(R, g);
        bc[R.i0 + g] = s;
        xc[R.i0 + g] = R.omc[g] * s;
    }
}

__device__ void fast_up(const Shared &sh, const View R, const double *x, double *xf) {
    const int tid = threadIdx.x;
    double *const xg = at_d(sh.xg);
    for (int e = tid; e < R.ents; e += kNT) xg[e] = x[R.col[e]];
    for (int k = tid; k < R.nrow; k += kNT) R.res[k] = x[R.id[k]];
    const int nm = R.mst[R.nrow];
    for (int q = tid; q < nm; q += kNT) R.mx[q] = xf[R.mem[q]];
    __syncthreads();
    for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
        const int k = ok ? R.ord[t] : 0;
        const double xi = R.res[k];
        double s = 0.0;
        if (ok) s = row_sum(R, k, sub, xg, sub ? 0.0 : R.bo[k] - R.dg[k] * xi);
        s = lanes_total(s, R.lg);
        if (ok && sub == 0) {
            const double val = xi + R.om[k] * s;
            for (int q = R.mst[k]; q < R.mst[k + 1]; ++q) xf[R.mem[q]] = R.mx[q] + val;
        }
    });
}

__device__ void fast_top(const Shared &sh, const View R, const double *x, double *z, double &rz, double &zq) {
    const int tid = threadIdx.x;
    double *const xg = at_d(sh.xg), *const zo = at_d(sh.zo);
    const double *const ro = at_d(sh.ro), *const qo = at_d(sh.qo);
    for (int e = tid; e < R.ents; e += kNT) xg[e] = x[R.col[e]];
    for (int k = tid; k < R.nrow; k += kNT) R.res[k] = x[R.id[k]];
    __syncthreads();
    for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
        const int k = ok ? R.ord[t] : 0;
        const double xi = R.res[k], ri = ro[k];
        double s = 0.0;
        if (ok) s = row_sum(R, k, sub, xg, sub ? 0.0 : ri - R.dg[k] * xi);
        s = lanes_total(s, R.lg);
        if (ok && sub == 0) {
            const double zi = xi + R.om[k] * s;
            zo[k] = zi;
            z[R.id[k]] = zi;
            rz += zi * ri;
            zq += zi * qo[k];
        }
    });
}

// yq (or null): gets om q, for fast_first.
__device__ void fast_product(const Shared &sh, const View R, const double *z, const double *pold, double beta, double *p,
                             double *yq, double &pq) {
    const int tid = threadIdx.x;
    double *const xg = at_d(sh.xg), *const po = at_d(sh.po), *const qo = at_d(sh.qo);
    const double *const zo = at_d(sh.zo);
    for (int e = tid; e < R.ents; e += kNT) {
        const int c = R.col[e];
        xg[e] = z[c] + beta * pold[c];
    }
    __syncthreads();
    for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
        const int k = ok ? R.ord[t] : 0;
        const double s = lanes_total(ok ? row_sum(R, k, sub, xg, 0.0) : 0.0, R.lg);
        if (ok && sub == 0) {
            const double pi = zo[k] + beta * po[k];
            po[k] = pi;
            p[R.id[k]] = pi;
            const double qi = R.dg[k] * pi - s;
            qo[k] = qi;
            if (yq) yq[R.id[k]] = R.om[k] * qi;
            pq += pi * qi;
        }
    });
}

// The step of the conjugate gradients and the finest level's way down in one
// pass: the neighbours' new smoothed values are xr - alpha yq, with xr = om r
// and yq = om q of before (the owner's own differs from that in its last bits
// at most, and only the preconditioner sees it).  A pass and a grid barrier
// less per iteration: a step at 96^2 82.1 ms instead of 85.2, at 320^2 502 instead
// of 531.
__device__ void fast_first(const Shared &sh, const View R, const double *xr, const double *yq, double alpha, double *xrn,
                           double *x, double *bc, double *xc, unsigned long long &mx) {
    const int tid = threadIdx.x;
    double *const xg = at_d(sh.xg), *const ro = at_d(sh.ro), *const dd = at_d(sh.dd);
    const double *const qo = at_d(sh.qo), *const po = at_d(sh.po), *const ibo = at_d(sh.ibo);
    for (int e = tid; e < R.ents; e += kNT) {
        const int c = R.col[e];
        xg[e] = xr[c] - alpha * yq[c];
    }
    for (int k = tid; k < R.nrow; k += kNT) {
        dd[k] += alpha * po[k];
        const double r = ro[k] - alpha * qo[k], v = R.om[k] * r;
        ro[k] = r;
        R.bo[k] = r;
        R.res[k] = v;
        xrn[R.id[k]] = v;
        x[R.id[k]] = v;
        mx = max_bits(mx, bits_of(fabs(r) * ibo[k]));
    }
    __syncthreads();
    for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
        const int k = ok ? R.ord[t] : 0;
        const bool in = ok && k < R.nmem;
        double s = 0.0;
        if (in) s = row_sum(R, k, sub, xg, sub ? 0.0 : R.bo[k] - R.dg[k] * R.res[k]);
        s = lanes_total(s, R.lg);
        if (in && sub == 0) R.res[k] = s;
    });
    __syncthreads();
    for (int g = tid; g < R.ngrp; g += kNT) {
        const double s = group_sum(R, g);
        bc[R.i0 + g] = s;
        xc[R.i0 + g] = R.omc[g] * s;
    }
}

// ---------------------------------------------------------------- the first cluster's levels

// The values of a spread level's entries into xs, of its rows into res and (with
// b) their right-hand sides into bo.
__device__ __forceinline__ void gather(const View &R, double *xs, bool with_b) {
    const int most = max(R.ents, R.nrow);
    for (int i = threadIdx.x; i < most; i += kNT) {
        const bool e = i < R.ents, k = i < R.nrow;
        const unsigned a = k ? R.xa[i] : 0;
        const double ve = e ? load_remote(static_cast<unsigned>(R.col[i])) : 0.0;
        const double vk = k ? load_remote(a) : 0.0;
        const double vb = k && with_b ? load_remote(a + R.db) : 0.0;
        if (e) xs[i] = ve;
        if (k) {
            R.res[i] = vk;
            if (with_b) R.bo[i] = vb;
        }
    }
}

// Levels t0 .. nlev - 1; on entry x of t0 holds om b (spread, or in every copy)
// and bo of its rows their b.  On return res of the block's rows at t0 is that
// level's result (a copied t0: of all rows, in every block).
__device__ void tier_cycle(const Shared &sh, unsigned rank, unsigned nr) {
    const int tid = threadIdx.x, t0 = sh.t0, tr = sh.tr, t1 = sh.nlev - 1;
    double *const xs = at_d(sh.xs);
    for (int t = t0; t < tr; ++t) {  // spread levels down
        const View R = view(sh.lev[t]);
        double *const xc = at_d(sh.lev[t + 1].x);
        const unsigned dc = sh.lev[t + 1].db;
        double *const bc = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(xc) + dc);
        gather(R, xs, t > t0);
        __syncthreads();
        for_rows(R.nrow, R.lg, [&](bool ok, int sub, int q) {
            const int k = ok ? R.ord[q] : 0;
            const bool in = ok && k < R.nmem;
            double s = 0.0;
            if (in) s = row_sum(R, k, sub, xs, sub ? 0.0 : R.bo[k] - R.dg[k] * R.res[k]);
            s = lanes_total(s, R.lg);
            if (in && sub == 0) R.res[k] = s;
        });
        __syncthreads();
        for (int g = tid; g < R.ngrp; g += kNT) {
            const double s = group_sum(R, g), x = s * R.omc[g];
            if (t + 1 < tr) {  // this block's aggregates are its range of the next level's nodes
                bc[g] = s;
                xc[g] = x;
            } else {
                store_all(bc + R.i0 + g, s, nr);
                store_all(xc + R.i0 + g, x, nr);
            }
        }
        cluster_sync();
    }
    for (int t = tr; t < t1; ++t) {  // copied levels down
        const View R = view(sh.lev[t]);
        const double *const b = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(R.x) + R.db);
        double *const xc = at_d(sh.lev[t + 1].x);
        double *const bc = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(xc) + sh.lev[t + 1].db);
        for_rows(R.nrow, R.lg, [&](bool ok, int sub, int q) {
            const int k = ok ? R.ord[q] : 0;
            const bool in = ok && k < R.nmem;
            double s = 0.0;
            if (in) {
                const int i = R.id[k];
                s = copy_sum(R, k, sub, R.x, sub ? 0.0 : b[i] - R.dg[k] * R.x[i]);
            }
            s = lanes_total(s, R.lg);
            if (in && sub == 0) R.res[k] = s;
        });
        __syncthreads();
        for (int g = tid; g < R.ngrp; g += kNT) {
            const double s = group_sum(R, g);
            bc[g] = s;
            xc[g] = s * R.omc[g];
        }
        __syncthreads();
    }
    {  // the coarsest level, copied
        const View Z = view(sh.lev[t1]);
        const double *const b = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(Z.x) + Z.db);
        if (sh.dense) {
            const double *const inv = at_d(sh.inv);
            // four lanes per row, two chains each
            for_items<4>(Z.n, [&](bool ok, int sub, int k) {
                double s0 = 0.0, s1 = 0.0;
                if (ok)
                    for (int j = sub; j < Z.n; j += 8) {
                        s0 += inv[k * kDense + j] * b[j];
                        if (j + 4 < Z.n) s1 += inv[k * kDense + j + 4] * b[j + 4];
                    }
                const double s = lanes_sum<4>(s0 + s1);
                if (ok && sub == 0) Z.res[k] = s;
            });
            __syncthreads();
        } else {
            double *const alt = at_d(sh.alt);
            for (int s = 0; s < sh.sweeps; ++s) {
                const double *x = (s & 1) ? alt : Z.x;
                double *xo = (s & 1) ? Z.x : alt;
                for_rows(Z.nrow, Z.lg, [&](bool ok, int sub, int k) {
                    double v = 0.0;
                    if (ok) v = copy_sum(Z, k, sub, x, sub ? 0.0 : b[k] - Z.dg[k] * x[k]);
                    v = lanes_total(v, Z.lg);
                    if (ok && sub == 0) {
                        const double val = x[k] + Z.om[k] * v;
                        Z.res[k] = val;
                        xo[k] = val;
                    }
                });
                __syncthreads();
            }
        }
    }
    for (int t = t1; t >= tr; --t) {  // copied levels up
        const View R = view(sh.lev[t]);
        if (t < t1) {
            const double *const b = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(R.x) + R.db);
            for_rows(R.nrow, R.lg, [&](bool ok, int sub, int q) {
                const int k = ok ? R.ord[q] : 0;
                const int i = R.id[k];
                const double xi = R.x[i];
                double s = 0.0;
                if (ok) s = copy_sum(R, k, sub, R.x, sub ? 0.0 : b[i] - R.dg[k] * xi);
                s = lanes_total(s, R.lg);
                if (ok && sub == 0) R.res[k] = xi + R.om[k] * s;
            });
            __syncthreads();  // the results are read by other threads than formed them
        }
        if (t == t0) return;
        const Rows &F = sh.lev[t - 1];
        double *const xf = at_d(F.x);
        if (t > tr) {
            for (int k = tid; k < R.nrow; k += kNT) {
                const double val = R.res[k];
                for (int q = R.mst[k]; q < R.mst[k + 1]; ++q) xf[R.mem[q]] += val;
            }
            __syncthreads();
        } else {  // into this block's range of the spread level
            int c0, c1;
            chunk(F.n, rank, nr, c0, c1);
            for (int k = tid; k < R.nrow; k += kNT) {
                const double val = R.res[k];
                for (int q = R.mst[k]; q < R.mst[k + 1]; ++q) {
                    const int i = R.mem[q];
                    if (i >= c0 && i < c1) xf[i - c0] += val;
                }
            }
            cluster_sync();
        }
    }
    for (int t = tr - 1; t >= t0; --t) {  // spread levels up
        const View R = view(sh.lev[t]);
        if (t > t0) {
            const int nm = R.mst[R.nrow];
            for (int q = tid; q < nm; q += kNT) R.mx[q] = load_remote(static_cast<unsigned>(R.mem[q]));
        }
        gather(R, xs, false);
        __syncthreads();
        for_rows(R.nrow, R.lg, [&](bool ok, int sub, int q) {
            const int k = ok ? R.ord[q] : 0;
            const double xi = R.res[k];
            double s = 0.0;
            if (ok) s = row_sum(R, k, sub, xs, sub ? 0.0 : R.bo[k] - R.dg[k] * xi);
            s = lanes_total(s, R.lg);
            if (ok && sub == 0) {
                const double val = xi + R.om[k] * s;
                if (t > t0)
                    for (int i = R.mst[k]; i < R.mst[k + 1]; ++i)
                        store_remote(static_cast<unsigned>(R.mem[i]), R.mx[i] + val);
                else
                    R.res[k] = val;
            }
        });
        if (t > t0) cluster_sync();
        else __syncthreads();
    }
}

// ---------------------------------------------------------------- the solve

// The right-hand side and the start's residual at row (id, its entries), in the
// sign-flipped unknowns (+1 rows, -1 columns); LPR lanes share it.
template <int LPR>
__device__ double start_residual(const PcgArgs &a, const HierView &v, int which, int id, int sub) {
    double s = 0.0;
    if (a.schur) {
        for (int64_t q = a.col_ptr[id] + sub; q < a.col_ptr[id + 1]; q += LPR) {
            const int32_t i = a.csc_row[q];
            s += a.a2c[q] * (a.rhs[i] / a.diag[i]);
        }
        if (sub == 0) s -= a.rhs[a.nc + id];
    } else if (sub == 0) {
        s = id < a.nc ? a.rhs[id] : -a.rhs[id];
    }
    if (which) {
        const int64_t e0 = v.rs[id];
        const int len = v.rl[id];
        for (int e = sub; e < len; e += LPR) s += v.ew[e0 + e] * a.d[v.ecol[e0 + e]];
        if (sub == 0) s -= v.dg[id] * a.d[id];
    }
    return lanes_sum<LPR>(s);
}

__device__ __forceinline__ double inverse_target(const PcgArgs &a, int id) {
    return 1.0 / (a.schur ? a.volphi[id] : (id < a.nc ? a.b_row[id] : a.volphi[id - a.nc]));
}

// One thread: alpha from the product's sum.
__device__ __forceinline__ void set_alpha(Shared &sh, double pq) {
    sh.conv = pq > 0.0 ? 0 : 1;
    sh.alpha = pq > 0.0 ? sh.rz / pq : 0.0;
}

// One thread: beta and the stopping test from z.r, z.q and the largest scaled residual.
__device__ __forceinline__ void set_beta(Shared &sh, double trz, double tres) {
    const double rz = sh.out[0], zq = sh.out[1], mx = sh.out[2];
    // z.(r - r_old) = -alpha z.q: the flexible (Polak-Ribiere) beta
    const double be = -sh.alpha * zq * sh.inv_rz;
    sh.beta = be > 0.0 ? be : 0.0;
    sh.rz = rz;
    sh.res_max = mx;
    if ((rz <= trz && mx <= tres) || !(rz > 0.0)) sh.conv = 1;
}

// 1 / (z.r) for the next beta, by a thread that nothing waits for (an FP64
// division takes ~600 clocks).
__device__ __forceinline__ void invert_rz(Shared &sh) {
    if (threadIdx.x == kNT - 32) sh.inv_rz = sh.rz > 0.0 ? 1.0 / sh.rz : 0.0;
}

// A system solved by one cluster: every level in its blocks' shared memory (the
// finest one spread).  Returns the iterations.
__device__ int solve_small(const PcgArgs &a, Shared &sh, unsigned rank, unsigned nr, int which, double trz, double tres,
                           int cap) {
    const HierView &v = a.v;
    const View R = view(sh.lev[0]);
    const int tid = threadIdx.x;
    double *const ro = at_d(sh.ro), *const dd = at_d(sh.dd), *const qo = at_d(sh.qo), *const po = at_d(sh.po);
    double *const zo = at_d(sh.zo), *const ibo = at_d(sh.ibo), *const xs = at_d(sh.xs), *const dots = at_d(sh.dots);
    // z and the two directions lie like x: an address of x plus these distances
    const int cx = (R.n + static_cast<int>(nr) - 1) / static_cast<int>(nr);
    const unsigned dz = sh.zv - sh.lev[0].x, dp = sh.pv - sh.lev[0].x;
    const unsigned pstep = static_cast<unsigned>(cx) * 8u;
    for_items<8>(R.nrow, [&](bool ok, int sub, int k) {
        const int id = ok ? R.id[k] : 0;
        const double s = start_residual<8>(a, v, which, id, sub);
        if (ok && sub == 0) {
            const double r = a.vcycle ? a.r[id] : s;
            ro[k] = r;
            dd[k] = which ? a.d[id] : 0.0;
            qo[k] = 0.0;
            po[k] = 0.0;
            ibo[k] = inverse_target(a, id);
            store_remote(R.xa[k], R.om[k] * r);
            store_remote(R.xa[k] + dp, 0.0);
        }
    });
    cluster_sync();
    int it = 0;
    unsigned long long mx = 0;
    for (;;) {
        tier_cycle(sh, rank, nr);
        // z is res of the own rows
        double rz = 0.0, zq = 0.0;
        for (int k = tid; k < R.nrow; k += kNT) {
            const double z = R.res[k];
            zo[k] = z;
            store_remote(R.xa[k] + dz, z);
            rz += z * ro[k];
            zq += z * qo[k];
        }
        block_partials(sh, 3, R.nrow, rz, zq, mx);
        if (tid < 3) store_all(dots + tid * 16 + rank, sh.out[tid], nr);
        cluster_sync();
        block_totals(sh, dots, 16, 3, nr);
        if (tid == 0) {
            if (it == 0) {
                sh.rz = sh.out[0];
                sh.beta = 0.0;
                sh.conv = sh.out[0] == 0.0 ? 1 : 0;
            } else {
                set_beta(sh, trz, tres);
            }
        }
        __syncthreads();
        if (sh.conv || it >= cap || a.vcycle) break;
        ++it;
        invert_rz(sh);
        const double beta = sh.beta;
        const unsigned old = dp + ((it + 1) & 1) * pstep, now = dp + (it & 1) * pstep;
        for (int e = tid; e < R.ents; e += kNT) {
            const unsigned c = static_cast<unsigned>(R.col[e]);
            const double z = load_remote(c + dz), p = load_remote(c + old);
            xs[e] = z + beta * p;
        }
        __syncthreads();
        double pq = 0.0;
        for_rows(R.nrow, R.lg, [&](bool ok, int sub, int t) {
            const int k = ok ? R.ord[t] : 0;
            const double s = lanes_total(ok ? row_sum(R, k, sub, xs, 0.0) : 0.0, R.lg);
            if (ok && sub == 0) {
                const double p = zo[k] + beta * po[k];
                po[k] = p;
                store_remote(R.xa[k] + now, p);
                const double q = R.dg[k] * p - s;
                qo[k] = q;
                pq += p * q;
            }
        });
        block_partials(sh, 1, R.nrow << R.lg, pq, 0.0, 0);
        if (tid == 0) store_all(dots + 48 + rank, sh.out[0], nr);
        cluster_sync();
        block_totals(sh, dots + 48, 16, 1, nr);
        if (tid == 0) set_alpha(sh, sh.out[0]);
        __syncthreads();
        const double alpha = sh.alpha;
        mx = 0;
        for (int k = tid; k < R.nrow; k += kNT) {
            const double r = ro[k] - alpha * qo[k];
            store_remote(R.xa[k], R.om[k] * r);
            ro[k] = r;
            dd[k] += alpha * po[k];
            mx = max_bits(mx, bits_of(fabs(r) * ibo[k]));
        }
        cluster_sync();
    }
    for (int k = tid; k < R.nrow; k += kNT) {
        a.d[R.id[k]] = dd[k];
        a.r[R.id[k]] = ro[k];
    }
    return it;
}

// One V-cycle across the grid; x of the finest level holds om r on entry, alt is
// a free vector of its size; first = 1: level 0's way down is done.  This
// thread's parts of z.r, z.q.
template <class Bar>
__device__ bool grid_cycle(const PcgArgs &a, Shared &sh, Bar &bar, int first, double *alt, double &rz,
                                        double &zq) {
    const HierView &v = a.v;
    const int nlev = sh.nlev, t0 = sh.t0;
    const int nd = t0 < nlev ? t0 : nlev - 1;  // shared levels that are aggregated
    for (int l = first; l < nd; ++l) {
        const Rows &R = sh.lev[l];
        double *bc = v.b + (R.noff + R.n), *xc = v.x + (R.noff + R.n);
        if (R.here == 1)
            fast_down(sh, view(R), l ? v.b + R.noff : nullptr, v.x + R.noff, bc, xc);
        else
            WITH_LANES(R.lprg, R.here, (general_down<LPR, HERE>(v, R, l ? v.b + R.noff : a.r, v.x + R.noff, bc, xc)));
        if (!bar.sync()) return false;
    }
    if (t0 < nlev) {
        const unsigned nr = cluster_size(), rank = blockIdx.x;
        if (rank < nr) {
            const View T = view(sh.lev[t0]);
            const bool spread = sh.lev[t0].kind == kSpread;
            const double *x = v.x + sh.lev[t0].noff, *bl = v.b + sh.lev[t0].noff;
            double *xf = v.x + sh.lev[t0 - 1].noff;
            int c0, c1, k0 = 0, k1 = T.nrow;
            if (spread) {
                chunk(T.n, rank, nr, c0, c1);
                for (int i = c0 + threadIdx.x; i < c1; i += kNT) T.x[i - c0] = x[i];
                for (int k = threadIdx.x; k < T.nrow; k += kNT) T.bo[k] = bl[T.id[k]];
                const int nm = T.mst[T.nrow];
                for (int q = threadIdx.x; q < nm; q += kNT) T.mx[q] = xf[T.mem[q]];
                cluster_sync();
            } else {
                chunk(T.nrow, rank, nr, k0, k1);  // every block has all results: each prolongs some
                double *const b = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(T.x) + T.db);
                for (int i = threadIdx.x; i < T.n; i += kNT) {
                    T.x[i] = x[i];
                    b[i] = bl[i];
                }
                __syncthreads();
            }
            tier_cycle(sh, rank, nr);
            for (int k = k0 + threadIdx.x; k < k1; k += kNT)
                for (int q = T.mst[k]; q < T.mst[k + 1]; ++q) {
                    double *to = xf + T.mem[q];
                    *to = (spread ? T.mx[q] : *to) + T.res[k];
                }
        }
        if (!bar.sync()) return false;
    } else {
        const Rows &R = sh.lev[nlev - 1];
        double *x = v.x + R.noff;
        const double *bl = nlev > 1 ? v.b + R.noff : a.r;
        if (sh.dense && nlev == 1) {  // a finest level of at most kDense nodes
            for (int k = threadIdx.x; k < R.nrow; k += kNT) {
                double s = 0.0;
                for (int j = 0; j < R.n; ++j) s += v.H->inv[(R.i0 + k) * kDense + j] * bl[j];
                x[R.i0 + k] = s;
            }
            if (!bar.sync()) return false;
        } else {
            for (int k = 0; k < sh.sweeps; ++k) {
                WITH_LANES(R.lpr, R.here, (general_sweep<LPR, HERE>(v, R, bl, (k & 1) ? alt : x, (k & 1) ? x : alt)));
                if (!bar.sync()) return false;
            }
        }
        if (nlev == 1) {
            for (int k = threadIdx.x; k < R.nrow; k += kNT) {
                const int i = R.i0 + k;
                const double zi = x[i];
                a.z[i] = zi;
                rz += zi * a.r[i];
                zq += zi * a.q[i];
            }
            return true;
        }
        const int64_t fine = sh.lev[nlev - 2].noff;
        for (int k = threadIdx.x; k < R.nrow; k += kNT)
            prolong(v, R.noff, fine, R.i0 + k, x[R.i0 + k], 0, 1, v.x + fine);
        if (!bar.sync()) return false;
    }
    for (int l = nd - 1; l > 0; --l) {
        const Rows &R = sh.lev[l];
        const int64_t fine = sh.lev[l - 1].noff;
        if (R.here == 1)
            fast_up(sh, view(R), v.x + R.noff, v.x + fine);
        else
            WITH_LANES(R.lpr, R.here, (general_up<LPR, HERE>(v, R, v.b + R.noff, v.x + R.noff, fine, v.x + fine)));
        if (!bar.sync()) return false;
    }
    const Rows &R = sh.lev[0];
    if (R.here == 1)
        fast_top(sh, view(R), v.x + 0, a.z, rz, zq);
    else
        WITH_LANES(R.lpr, R.here, (general_top<LPR, HERE>(v, R, a.r, a.q, v.x + 0, a.z, rz, zq)));
    return true;
}

// A system shared by all blocks.  Returns the iterations, -1 when a barrier failed.
template <class Bar>
__device__ int solve_grid_wide(const PcgArgs &a, Shared &sh, Bar &bar, int which, double trz, double tres, int cap) {
    const HierView &v = a.v;
    Hier *H = v.H;
    const Rows &R = sh.lev[0];
    const View O = view(R);  // with the rows in shared memory
    double *const ro = at_d(sh.ro), *const dd = at_d(sh.dd), *const qo = at_d(sh.qo), *const po = at_d(sh.po);
    double *const ibo = at_d(sh.ibo), *const xg = at_d(sh.xg);
    const unsigned b = blockIdx.x, nb = gridDim.x;
    const int tid = threadIdx.x;
    double *pbuf[2] = {a.p0, a.p1};
    const bool here = R.here == 1;
    // rows of every block in shared memory: the vectors there leave a.ib, a.r (om r, in turns)
    // and a.q (om q) free for fast_first
    const bool fused = a.e0 <= kFuseEntries * nb;
    const bool lean = fused && sh.nlev > 1 && !a.vcycle && *reinterpret_cast<volatile int *>(&H->general) == 0;
    double *xr[2] = {a.ib, a.r};
    for_items<8>(R.nrow, [&](bool ok, int sub, int k) {
        int id = 0;
        if (ok) id = here ? O.id[k] : row_id(v, R, k);
        const double s = start_residual<8>(a, v, which, id, sub);
        if (ok && sub == 0) {
            const double r = a.vcycle ? a.r[id] : s, ib = inverse_target(a, id);
            a.p0[id] = 0.0;
            if (here) {
                ro[k] = r;
                dd[k] = which ? a.d[id] : 0.0;
                qo[k] = 0.0;
                po[k] = 0.0;
                ibo[k] = ib;
            } else {
                if (!a.vcycle) a.r[id] = r;
                a.q[id] = 0.0;
                a.ib[id] = ib;
            }
            v.x[id] = v.om[id] * r;
            if (lean) a.ib[id] = v.om[id] * r;
        }
    });
    if (!bar.sync()) return -1;
    if (!here && !which && !a.vcycle)  // after the barrier: other rows' starts may read d
        for (int k = tid; k < R.nrow; k += kNT) a.d[row_id(v, R, k)] = 0.0;
    int it = 0;
    unsigned long long mx = 0;
    for (;;) {
        double rz = 0.0, zq = 0.0;
        if (!grid_cycle(a, sh, bar, lean && it ? 1 : 0, pbuf[(it + 1) & 1], rz, zq)) return -1;
        if (a.vcycle) return 0;
        block_partials(sh, 3, here ? R.nrow << R.lg : kNT, rz, zq, mx);
        if (tid < 3) H->part[1 + tid][b] = sh.out[tid];
        if (!bar.sync()) return -1;
        block_totals(sh, H->part[1], kMaxCtas, 3, nb);
        if (tid == 0) {
            if (it == 0) {
                sh.rz = sh.out[0];
                sh.beta = 0.0;
                sh.conv = sh.out[0] == 0.0 ? 1 : 0;
            } else {
                set_beta(sh, trz, tres);
            }
        }
        __syncthreads();
        if (sh.conv || it >= cap) break;
        ++it;
        invert_rz(sh);
        const double beta = sh.beta;
        const double *pold = pbuf[(it + 1) & 1];
        double *pn = pbuf[it & 1];
        double pq = 0.0;
        if (!fused) {  // grid-uniform
            for (int k = tid; k < R.nrow; k += kNT) {
                const int i = here ? O.id[k] : row_id(v, R, k);
                pn[i] = a.z[i] + beta * pold[i];
            }
            if (!bar.sync()) return -1;
            if (here) {
                for (int e = tid; e < O.ents; e += kNT) xg[e] = pn[O.col[e]];
                __syncthreads();
                for_rows(O.nrow, O.lg, [&](bool ok, int sub, int t) {
                    const int k = ok ? O.ord[t] : 0;
                    const double s = lanes_total(ok ? row_sum(O, k, sub, xg, 0.0) : 0.0, O.lg);
                    if (ok && sub == 0) {
                        const double pi = pn[O.id[k]], qi = O.dg[k] * pi - s;
                        po[k] = pi;
                        qo[k] = qi;
                        pq += pi * qi;
                    }
                });
            } else {
                WITH_LANES(R.lpr, R.here, (general_product<LPR, HERE, false>(v, R, a.z, pold, beta, pn, a.q, pq)));
            }
        } else if (here) {
            fast_product(sh, O, a.z, pold, beta, pn, lean ? a.q : nullptr, pq);
        } else {
            WITH_LANES(R.lpr, R.here, (general_product<LPR, HERE, true>(v, R, a.z, pold, beta, pn, a.q, pq)));
        }
        block_partials(sh, 1, here ? R.nrow << R.lg : kNT, pq, 0.0, 0);
        if (tid == 0) H->part[0][b] = sh.out[0];
        if (!bar.sync()) return -1;
        block_totals(sh, H->part[0], kMaxCtas, 1, nb);
        if (tid == 0) set_alpha(sh, sh.out[0]);
        __syncthreads();
        const double alpha = sh.alpha;
        mx = 0;
        if (lean) {
            const int64_t c = R.noff + R.n;  // the next level's nodes
            fast_first(sh, O, xr[(it + 1) & 1], a.q, alpha, xr[it & 1], v.x + 0, v.b + c, v.x + c, mx);
        }
        for (int k = lean ? R.nrow : tid; k < R.nrow; k += kNT) {
            if (here) {
                dd[k] += alpha * po[k];
                const double r = ro[k] - alpha * qo[k];
                ro[k] = r;
                v.x[O.id[k]] = O.om[k] * r;
                mx = max_bits(mx, bits_of(fabs(r) * ibo[k]));
            } else {
                const int i = row_id(v, R, k);
                a.d[i] += alpha * pn[i];
                const double r = a.r[i] - alpha * a.q[i];
                a.r[i] = r;
                v.x[i] = v.om[i] * r;
                mx = max_bits(mx, bits_of(fabs(r) * a.ib[i]));
            }
        }
        if (!bar.sync()) return -1;
    }
    if (here)
        for (int k = tid; k < R.nrow; k += kNT) {
            a.d[O.id[k]] = dd[k];
            a.r[O.id[k]] = ro[k];
        }
    return it;
}

// The finest level's own vectors, n values each, at f.
__device__ __forceinline__ void own_vectors(Shared &sh, unsigned f, int n) {
    const unsigned s = 8u * static_cast<unsigned>(n);
    sh.ro = f;
    sh.dd = f + s;
    sh.qo = f + 2 * s;
    sh.po = f + 3 * s;
    sh.zo = f + 4 * s;
    sh.ibo = f + 5 * s;
}

// ONE: the grid is one cluster, for a small system.
template <bool ONE> __global__ void __launch_bounds__(kSolveThreads, 1) k_pcg(const __grid_constant__ PcgArgs a) {
    __shared__ Shared sh;
    const HierView &v = a.v;
    Hier *H = v.H;
    const unsigned b = blockIdx.x, nb = gridDim.x;
    const unsigned rank = cluster_rank(), nr = cluster_size();
    const int tid = threadIdx.x;
    const IpArgs &ip = a.ip;
    GridBarT<ONE> bar(&H->bar[a.vcycle ? 2 : 1], &ip.st->err, nb);
    // formed where it is used: held through the solves it costs a register too many
    auto end_of_block = [&]() { return ClusterEnd{&v.H->left[a.vcycle ? 1 : 0][blockIdx.x / cluster_size()], cluster_size()}; };
    // an earlier barrier failed: nothing here can be relied on; or the iterations have ended
    if (__syncthreads_or(ip.st->err | (a.vcycle ? 0 : ip.st->stop))) {
        end_of_block().done();
        return;
    }
    int *const notier = &H->notier[a.vcycle ? 1 : 0];
    __shared__ IpShared ips;
    int64_t r0, r1;
    ip_range(ip.nc, b, nb, r0, r1);
    const double mu = ip.st->mu, rp_max = ip.st->rp_max;
    int cg = ip.st->cg;
    const int done = ip.st->it;
    if (!a.vcycle) {
        if (b == 0 && tid == 0) H->bar[0] = 0;  // for the next build
        ip_q<kIpLanes>(ip, r0, r1, 0, 0.0);
    }

    // the levels: t0 is the first of the first cluster's (nlev: none), tr the first copied one
    if (tid == 0) {
        const int nlev = H->nlev;
        int t0 = nlev;
        for (int l = nlev - 1; l >= (ONE ? 0 : 1); --l) {
            if (!ONE && (H->L[l].nnz > kTierEntries || H->L[l].n > kTierNodes)) break;
            t0 = l;
        }
        if (ONE && nlev == 1) t0 = nlev;
        int tr = nlev - 1;
        while (tr - 1 > t0 && H->L[tr - 1].n <= kCopyNodes && H->L[tr - 1].nnz <= kCopyEntries) --tr;
        sh.nlev = nlev;
        sh.dense = H->dense;
        sh.sweeps = H->sweeps;
        sh.t0 = t0;
        sh.tr = tr;
        for (int l = 0; l < nlev; ++l) sh.lev[l].kind = l < t0 ? kGrid : (l < tr ? kSpread : kCopy);
    }
    __syncthreads();
    unsigned p = 0;
    const unsigned end = a.smem;
    bool ok = true;
    if (b < nr && sh.t0 < sh.nlev) {
        // the vectors first: they are at the same place in every block of the cluster
        size_t bytes = 2048 + sizeof(double) * kDense * (kDense + 1);
        for (int t = sh.t0; t < sh.nlev; ++t)
            bytes += 2 * (sh.lev[t].kind == kSpread ? (H->L[t].n + nr - 1) / nr : H->L[t].n) * sizeof(double) + 16;
        if (!sh.dense) bytes += sizeof(double) * H->L[sh.nlev - 1].n;
        const int cx = (a.n0 + static_cast<int>(nr) - 1) / static_cast<int>(nr);
        if (sh.t0 == 0) bytes += sizeof(double) * 3 * cx;
        ok = bytes <= a.smem;
        if (ok) {
            for (int t = sh.t0; t < sh.nlev; ++t) {
                const int n = H->L[t].n;
                const int len = sh.lev[t].kind == kSpread ? (n + static_cast<int>(nr) - 1) / static_cast<int>(nr) : n;
                const unsigned x = take_n<double>(p, 2 * len);
                if (tid == 0) {
                    sh.lev[t].x = x;
                    sh.lev[t].db = 8u * static_cast<unsigned>(len);
                }
            }
            const unsigned alt = take_n<double>(p, sh.dense ? 1 : H->L[sh.nlev - 1].n), dots = take_n<double>(p, 64);
            const unsigned zv = take_n<double>(p, sh.t0 == 0 ? 3 * cx : 1);
            const unsigned inv = take_n<double>(p, sh.dense ? kDense * kDense : 1);
            if (tid == 0) {
                sh.alt = alt;
                sh.dots = dots;
                sh.zv = zv;
                sh.pv = zv + 8u * static_cast<unsigned>(cx);
                sh.inv = inv;
            }
            __syncthreads();
            if (sh.dense)
                for (int i = tid; i < kDense * kDense; i += kNT) at_d(inv)[i] = H->inv[i];
        }
        // room is kept for the finest level's own vectors and a pass's gathered values
        int most = 0;
        for (int t = sh.nlev - 1; t >= sh.t0 && ok; --t) {
            ok = load_rows(v, sh, t, sh.lev[t].kind, static_cast<int>(rank), static_cast<int>(nr), p, end, 0, most);
            if (ok && sh.lev[t].kind == kSpread) most = max(most, sh.lev[t].ents);
        }
        if (ok && sh.t0 < sh.tr) {
            const int n = sh.t0 == 0 ? sh.lev[0].nrow : 0;
            if (static_cast<size_t>(end - p) < static_cast<size_t>(n) * 48 + static_cast<size_t>(most) * 8 + 128) {
                ok = false;
            } else {
                const unsigned f = take_n<double>(p, 6 * n), xs = take_n<double>(p, most);
                if (tid == 0) {
                    own_vectors(sh, f, n);
                    if (n > 0) sh.lev[0].bo = sh.ro;  // the finest level's right-hand side is the residual
                    sh.xs = xs;
                }
            }
        }
        __syncthreads();
        if (!ok && tid == 0) atomicExch(notier, 1);
    }
    bool go = bar.sync();
    if (go && *reinterpret_cast<volatile int *>(notier)) {  // grid-uniform
        if (tid == 0) sh.t0 = sh.nlev;
        p = 0;
        __syncthreads();
    }
    const bool alone = ONE && sh.t0 == 0;
    if (go && !alone) {
        // shared levels, the finest first; the gathered values of a pass go to the end of the arrays
        const int ns = sh.t0 < sh.nlev ? sh.t0 : sh.nlev;
        int most = 0;
        for (int l = 0; l < ns; ++l) {
            const bool coarsest = l == sh.nlev - 1;
            size_t own = 0;
            const unsigned before = p;
            if (l == 0 && !coarsest) {  // room for the finest level's own vectors
                const Seg g = H->L[0].grid || b == 0 ? v.seg[b] : Seg{};
                own = static_cast<size_t>(g.mlen + g.llen) * 48 + 128;
            }
            const bool got = !coarsest && load_rows(v, sh, l, kGrid, static_cast<int>(b), static_cast<int>(nb), p, end,
                                                    own, most) &&
                             (ONE ? sh.lev[l].here == 1 : sh.lev[l].here != 0);
            if (coarsest) {
                unsigned q = p;  // rows are read from global memory: only the description is wanted
                load_rows(v, sh, l, kGrid, static_cast<int>(b), static_cast<int>(nb), q, q, 1, 0);
            }
            if (got) {
                if (sh.lev[l].here == 1) most = max(most, sh.lev[l].ents);
                if (l == 0 && sh.lev[l].here == 1) {
                    const int n = sh.lev[0].nrow;
                    const unsigned f = take_n<double>(p, 6 * n);
                    if (tid == 0) own_vectors(sh, f, n);
                }
            } else {
                p = before;
                if (tid == 0) sh.lev[l].here = 0;
            }
            __syncthreads();
        }
        if (tid == 0) {
            sh.xg = p;
            if (!a.vcycle && sh.lev[0].here != 1) atomicExch(&H->general, 1);
        }
        __syncthreads();
    }

    if (go && a.vcycle) {
        go = (alone ? solve_small(a, sh, rank, nr, 0, 0.0, 0.0, 1) : solve_grid_wide(a, sh, bar, 0, 0.0, 0.0, 1)) >= 0;
    } else if (go) {
        ip_rhs<kIpLanes>(ip, r0, r1, 0, 0.0);
        go = bar.sync();
    }
    for (int corr = 0; corr < 2 && go && !a.vcycle; ++corr) {
        const SolveTol &tol = corr ? (mu <= a.tols.last_mu ? a.tols.last : a.tols.corrector) : a.tols.predictor;
        const double trz = tol.rz_rel * mu, tres = fmax(tol.res_rel * rp_max, tol.res_floor);
        const int cap = max(1, min(a.tols.max_iter, ip.max_cg - cg));
        const int it = alone ? solve_small(a, sh, rank, nr, corr, trz, tres, cap)
                             : solve_grid_wide(a, sh, bar, corr, trz, tres, cap);
        cg += it;
        go = it >= 0 && bar.sync();
        if (!go) break;
        // back to the unknowns of rows and columns
        if (a.schur)
            ip_items<kIpLanes>(r0, r1, [&](bool ok, int sub, int64_t i) {
                double s = 0.0;
                if (ok)
                    for (int64_t e = a.row_ptr[i] + sub; e < a.row_ptr[i + 1]; e += kIpLanes) s += a.a2[e] * a.d[a.col[e]];
                s = ip_lanes<kIpLanes>(s);
                if (ok && sub == 0) a.dy[i] = (a.rhs[i] + s) / a.diag[i];
                if (ok && sub == 1) a.dy[a.nc + i] = -a.d[i];
            });
        else
            for (int64_t i = r0 + tid; i < r1; i += kNT) {
                a.dy[i] = a.d[i];
                a.dy[a.nc + i] = -a.d[a.nc + i];
            }
        __syncthreads();
        go = ip_steps(ip, bar, ips, r0, r1, a.d + (a.schur ? 0 : a.nc), -1.0);
        if (go) go = corr ? ip_step(ip, bar, ips, r0, r1, cg, done + 1) : ip_corrector(ip, bar, ips, r0, r1) && bar.sync();
    }
    if (b == 0 && tid == 0 && !a.vcycle) {
        ip.st->levels = sh.nlev;
        ip.st->coarsest = H->L[sh.nlev - 1].n;
    }
    // no block leaves while another may still store into its shared memory
    ClusterEnd here = end_of_block();
    leave_cluster(here, !go);
}

// One damped-Jacobi sweep of the finest level (timing).
__global__ void k_level_sweep(HierView v, int n, const double *b, const double *x, double *xo) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t e0 = v.rs[i];
        const int len = v.rl[i];
        double s = v.dg[i] * x[i];
        for (int e = 0; e < len; ++e) s -= v.ew[e0 + e] * x[v.ecol[e0 + e]];
        xo[i] = x[i] + v.om[i] * (b[i] - s);
    }
}

// ---------------------------------------------------------------- host side

static PcgArgs pcg_args(bchar_mesh_t m) {
    Amg &A = m->amg;
    PcgArgs a{};
    a.v = hier_view(m);
    a.n0 = static_cast<int>(A.n0);
    a.e0 = A.e0;
    a.schur = A.schur ? 1 : 0;
    a.nc = m->nc;
    a.row_ptr = ptr<int64_t>(m->row_ptr);
    a.col_ptr = ptr<int64_t>(m->col_ptr);
    a.col = ptr<int32_t>(m->col);
    a.csc_row = ptr<int32_t>(m->csc_row);
    a.a2 = ptr<double>(m->a2);
    a.a2c = ptr<double>(m->a2c);
    a.diag = ptr<double>(m->diag);
    a.rhs = ptr<double>(m->rhs);
    a.dy = ptr<double>(m->cg_d);
    double *w = ptr<double>(A.vec);
    double **dst[] = {&a.d, &a.r, &a.p0, &a.p1, &a.q, &a.z, &a.ib};
    for (double **d : dst) {
        *d = w;
        w += A.n0;
    }
    a.b_row = ptr<double>(m->bloc);
    a.volphi = ptr<double>(m->volphi);
    return a;
}

static void launch_pcg(bchar_mesh_t m, PcgArgs &a) {
    const SolveShape s = solve_shape(m);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(s.grid);
    cfg.blockDim = dim3(kSolveThreads);
    a.smem = static_cast<unsigned>(s.small ? kSolveSmem : solve_smem_of(a.e0, s.grid));
    cfg.dynamicSmemBytes = a.smem;
    cfg.stream = m->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s.cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = s.small ? 1 : 2;  // one cluster is resident as a whole
    cudaLaunchKernelEx(&cfg, s.small ? k_pcg<true> : k_pcg<false>, a);
    ++m->launches;
}

void pcg_opt_in() {
    cudaFuncSetAttribute(k_pcg<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSolveSmem));
    cudaFuncSetAttribute(k_pcg<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSolveSmem));
    cudaFuncSetAttribute(k_pcg<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

SolveRoom solve_room() {
    SolveRoom r;
    int n = 0;
    r.blocks = kWideCluster;
    if (clusters_resident(k_pcg<false>, kWideCluster, kNT, kSolveSmem, &n) && n > 1) r.blocks = n * kWideCluster;
    r.small = clusters_resident(k_pcg<true>, kSmallCluster, kNT, kSolveSmem, &n) && n >= 1;
    return r;
}

void pcg_launch(bchar_mesh_t m, const IpArgs &ip, const SolveTols &tols) {
    PcgArgs a = pcg_args(m);
    a.ip = ip;
    a.tols = tols;
    launch_pcg(m, a);
}

void amg_vcycle_once(bchar_mesh_t m) {
    PcgArgs a = pcg_args(m);
    a.ip.st = ip_scalars(m);
    a.vcycle = 1;
    Hier *H = ptr<Hier>(m->amg.hier);
    cudaMemsetAsync(&H->bar[2], 0, sizeof(unsigned), m->stream);
    cudaMemsetAsync(&H->notier[1], 0, sizeof(int), m->stream);
    cudaMemsetAsync(H->left[1], 0, sizeof H->left[1], m->stream);
    launch_pcg(m, a);
}

void amg_smooth_once(bchar_mesh_t m) {
    const PcgArgs a = pcg_args(m);
    k_level_sweep<<<blocks_for(a.n0), kThreads, 0, m->stream>>>(a.v, a.n0, a.r, a.z, a.q);
    ++m->launches;
}

}  // namespace bchar
