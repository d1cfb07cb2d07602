// The aggregation-multigrid hierarchy of the minimisation's linear system,
// built by one cooperative kernel.
//
// The system is the symmetric M-matrix L = diag(ex) + graph Laplacian of
// weights w > 0 on the finest level's nodes (the columns of A once the rows are
// eliminated, schur.cu; or rows and columns), a level's operator being kept as
// (diagonal, weights): L = dg - W, dg_i = ex_i + sum_j w_ij.  The excess ex
// (the shift) is carried separately because it is down to ~1e-14 of the
// weights and differences of diagonals would cancel it away.
//
// The conditioning is poor on two counts: mesh-scale smooth modes, and weak
// links (near-tangent ball overlaps).  A cluster of nodes held to the rest only
// by weak links has a near-null mode (constant on the cluster); the coarse
// levels keep that mode only if no aggregate straddles the weak links.  So the
// aggregation follows strong links alone:
//   - an edge is strong when its weight is at least kStrength sqrt(d_i d_j);
//   - each level pairs every node with its top-ranked strong neighbour when the
//     choice is mutual (kHandshakes rounds, each among the nodes still
//     unpaired); a node left unpaired joins the aggregate of its top-ranked
//     neighbour when that edge carries kAttach of its diagonal, else stays single;
//   - a node whose off-diagonal weights sum to at most kDominant of its
//     diagonal (a constraint held by its shift) leaves the hierarchy: the
//     smoother alone reduces its error by about that ratio per sweep, and left
//     in, such nodes stall the coarsening.  Its edges to the nodes that stay are
//     carried into their coarse shift, so the coarse operator is the Galerkin
//     product P^T L P for the piecewise-constant P of the aggregates;
//   - coarsening stops at kDense nodes (that level's inverse is formed), when a
//     level would keep more than kStall of its remaining nodes, or when the
//     arrays are full.
// Neighbours are ranked by (binary exponent of the weight, symmetric hash of
// the edge): by the exact weight, the weights of smooth flows grow along the
// strong chains of the graph, every node points the same way and almost no
// choice is mutual.
//
// Why one kernel: a level takes about twenty-five dependent passes of a few
// microseconds; launched one by one, with the level sizes read back by the
// host, a build took 1.5 to 3 ms on meshes of 10^3 to 6 x 10^4 cells, and an
// interior point builds 15 to 75 of them.  Here seven passes per level run
// between grid barriers (pairing ranks fused with the attachment and leaving
// tests, the leader decisions evaluated in one pass from the ranks, one pass
// per coarse row instead of count and fill), the sizes stay on the device, and
// levels of at most kBlockEntries entries are built by block 0 alone between
// block barriers.  The arithmetic does not depend on where a row is stored
// (block shares of the entry arrays are claimed by an atomic cursor), and every
// sum runs in a fixed order: the hierarchy is deterministic.
#include <math.h>
#include <stddef.h>

#include "amg.cuh"
#include "device.cuh"
#include "gridbar.cuh"
#include "ip.cuh"

namespace bchar {

constexpr int kHandshakes = 2;        // matching rounds (four gave the same iteration counts)
constexpr double kStall = 0.9;        // stop coarsening when a level keeps this fraction of nodes
constexpr double kStrength = 0.1;     // strong edge: w_ij >= kStrength sqrt(d_i d_j)
constexpr double kAttach = 0.25;      // a leftover node follows an edge carrying this share of its diagonal
constexpr double kDominant = 0.25;    // a node leaves when its off-diagonal sum is this share of its diagonal
// Jacobi damping of rows with off-diagonal entries: on the eliminated system
// 0.7, 0.8, 0.9 took 2 595, 2 545, 2 676 iterations on a 128^2 stretched step and
// 827, 810, 839 on a porous 24^3 one; 1.0 and above does not converge.
constexpr double kOmega = 0.8;
constexpr int kLargeSweeps = 20;      // Jacobi sweeps of a coarsest level that is not solved by its inverse
constexpr int kDominantSweeps = 4;    // the same when all of its nodes are diagonally dominant

constexpr int kWarpRaw = 256;                          // entries of a coarse row merged by one warp
constexpr int kBlockRaw = kWarpRaw * (kBuildThreads / 32);  // by the whole block
constexpr size_t kBuildSmem = static_cast<size_t>(kBlockRaw) * (sizeof(unsigned long long) + sizeof(double));

struct BuildArgs {
    HierView v;
    int n0;          // nodes and entries of the finest level
    int64_t e0;
    int schur;       // 1: columns with the rows eliminated, 0: rows and columns
    int64_t nc;
    const int64_t *col_ptr;
    const int32_t *csc_row;
    const double *a2, *a2c, *diag, *exc;  // the bipartite system: weights by row and by column, 2 n_c diagonals and shifts
    const double *g, *t;                  // a2 / sqrt(diag_row) per entry; exc / diag per row
    const uint32_t *cs;                   // first contribution of each entry of the finest level
    const int2 *pair;                     // contributions: two entries of one row of A
    IpArgs ip;
    int same;                             // 1: the aggregates of the build before
    int32_t *best0, *best1, *partner, *att, *lead, *pos, *cnt, *cap;  // n0 each
};

__device__ __forceinline__ uint32_t edge_hash(int64_t i, int64_t j) {
    const uint64_t a = static_cast<uint64_t>(i < j ? i : j), b = static_cast<uint64_t>(i < j ? j : i);
    uint64_t x = (a * 0x9E3779B1ull + b * 0x85EBCA77ull) & 0xFFFFFFFFull;
    x ^= x >> 16;
    x = (x * 0x7FEB352Dull) & 0xFFFFFFFFull;
    x ^= x >> 15;
    x = (x * 0x846CA68Bull) & 0xFFFFFFFFull;
    x ^= x >> 16;
    return static_cast<uint32_t>(x);
}

// Rank of an edge: exponent field of the weight, then the hash.
__device__ __forceinline__ unsigned long long edge_rank(int i, int j, int hi) {
    return (static_cast<unsigned long long>(hi >> 20) << 32) | edge_hash(i, j);
}

// The high word of a positive double is monotone in it, and as an integer a
// piecewise linear log2 in units of 2^-20 (off by at most 0.086): the tests of
// the matching compare those, because a warp instruction of the FP64 pipe costs
// 19 clocks of the SM and an integer one a quarter of a clock.
__device__ __forceinline__ int high_word(double w) { return __double2hiint(w); }
constexpr int kStrengthHi = 3483294;  // -log2(kStrength) = 3.3219, in those units
constexpr int kAttachHi = 2 << 20;    // -log2(kAttach)
static_assert(kStrength == 0.1 && kAttach == 0.25, "the constants above follow them");
// Whether an edge of weight w is strong between diagonals di and dj, w >= kStrength
// sqrt(di dj); whether it carries kAttach of di.  The sum of two high words passes
// 2^31 from weights of 0.2 on (a mesh given in metres, or in cell widths): with 32
// bits a 96^2 step on a square of side 1 024 took 3.6 times the CG iterations.
__device__ __forceinline__ bool strong_edge(int w, int di, int dj) {
    return 2ll * w + 2 * kStrengthHi >= static_cast<long long>(di) + dj;
}
__device__ __forceinline__ bool carries_diagonal(int w, int di) {
    return static_cast<long long>(w) + kAttachHi >= di;
}

// The higher-ranked of (key, j) and (k2, j2); j < 0 is none; ties go to the smaller node.
__device__ __forceinline__ void take_higher(unsigned long long &key, int &j, unsigned long long k2, int j2) {
    if (j2 >= 0 && (j < 0 || k2 > key || (k2 == key && j2 < j))) {
        key = k2;
        j = j2;
    }
}

// Exclusive scan of one int per thread over the block (kBuildThreads); tmp: 33 ints of shared memory.
__device__ __forceinline__ int block_scan(int x, int *tmp, int &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = x;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();  // tmp may still be read from the previous call
    if (lane == 31) tmp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int t = tmp[lane], s = t;
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

__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// ---- a level's diagonals, one thread per row: the entries' weights are summed
// to the diagonal on top of the excess (base: what the row has of it so far), and
// the node is marked when it leaves the hierarchy (partner: -3, else -1).

__device__ __forceinline__ void finish_row(const HierView &v, int64_t k, double ex, int32_t *partner) {
    const int64_t e0 = v.rs[k];
    const int len = v.rl[k];
    double s = 0.0;
    for (int e = 0; e < len; ++e) s += v.ew[e0 + e];
    const double d = ex + s;
    v.ex[k] = ex;
    v.dg[k] = d;
    v.om[k] = (len == 0 ? 1.0 : kOmega) / d;
    *partner = len == 0 || ex >= (1.0 - kDominant) * d ? -3 : -1;
}

// ---- the finest level's weights (LPR lanes per row), then its diagonals

template <int LPR> __device__ void level0_values(const BuildArgs &a, int i0, int i1) {
    const int lane = threadIdx.x & 31, sub = lane % LPR;
    const HierView &v = a.v;
    for (int i = i0 + static_cast<int>(threadIdx.x) / LPR; i < i1; i += blockDim.x / LPR) {
        const int64_t e0 = v.rs[i];
        const int len = v.rl[i];
        if (a.schur) {
            for (int e = sub; e < len; e += LPR) {
                double w = 0.0;
                const uint32_t k1 = a.cs[e0 + e + 1];
                for (uint32_t k = a.cs[e0 + e]; k < k1; ++k) {
                    const int2 p = a.pair[k];
                    w += a.g[p.x] * a.g[p.y];
                }
                v.ew[e0 + e] = w;
            }
        } else {
            const bool row = i < a.nc;
            const int64_t src = row ? e0 : a.col_ptr[i - a.nc];  // the row entries come first, in CSR order
            for (int e = sub; e < len; e += LPR) v.ew[e0 + e] = row ? a.a2[src + e] : a.a2c[src + e];
        }
    }
    __syncthreads();
    for (int i = i0 + static_cast<int>(threadIdx.x); i < i1; i += blockDim.x) {
        double ex;
        if (a.schur) {
            ex = a.exc[a.nc + i];
            for (int64_t p = a.col_ptr[i]; p < a.col_ptr[i + 1]; ++p) ex += a.a2c[p] * a.t[a.csc_row[p]];
        } else {
            ex = a.exc[i];
        }
        finish_row(v, i, ex, &a.partner[i]);
    }
}

// ---- one matching round (LPR lanes per node of the level at node offset noff)

template <int LPR>
__device__ void rank_round(const BuildArgs &a, int64_t noff, int i0, int i1, int round, const int32_t *bprev,
                           int32_t *bcur) {
    const HierView &v = a.v;
    const int lane = threadIdx.x & 31, sub = lane % LPR;
    volatile int32_t *partner = a.partner;
    for (int r0 = i0 + static_cast<int>(threadIdx.x >> 5) * (32 / LPR); r0 < i1; r0 += blockDim.x / LPR) {
        const int i = r0 + lane / LPR;
        const bool ok = i < i1;
        unsigned long long key = 0, akey = 0;
        int bj = -1, aj = -1, mate = -3, wmax = 0, di = 0;
        if (ok) {
            di = high_word(v.dg[noff + i]);
            mate = partner[i];
            if (round > 0 && mate == -1) {  // did the previous round's choices meet?
                const int b = bprev[i];
                if (b >= 0 && bprev[b] == i) mate = b;
            }
            if (mate == -1) {
                const int64_t e0 = v.rs[noff + i];
                const int len = v.rl[noff + i];
                for (int e = sub; e < len; e += LPR) {
                    const int j = v.ecol[e0 + e];
                    const int w = high_word(v.ew[e0 + e]);
                    if (w <= 0) continue;
                    if (partner[j] != -1) continue;
                    if (round > 0) {
                        const int b = bprev[j];
                        if (b >= 0 && bprev[b] == j) continue;
                    }
                    const unsigned long long k = edge_rank(i, j, w);
                    if (round == 0) {
                        wmax = max(wmax, w);
                        take_higher(akey, aj, k, j);
                    }
                    if (strong_edge(w, di, high_word(v.dg[noff + j]))) take_higher(key, bj, k, j);
                }
            }
        }
        for (int o = LPR / 2; o > 0; o >>= 1) {
            take_higher(key, bj, __shfl_xor_sync(0xffffffffu, key, o), __shfl_xor_sync(0xffffffffu, bj, o));
            if (round == 0) {
                take_higher(akey, aj, __shfl_xor_sync(0xffffffffu, akey, o), __shfl_xor_sync(0xffffffffu, aj, o));
                wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
            }
        }
        if (ok && sub == 0) {
            bcur[i] = bj;
            if (round > 0) {
                partner[i] = mate;
            } else {
                // one-sided on purpose: a leaf hanging off a hub by an edge that is most of
                // its own diagonal but little of the hub's should follow the hub
                a.att[i] = (aj >= 0 && carries_diagonal(wmax, di)) ? aj : -1;
                a.cnt[i] = 0;
                a.cap[i] = 0;
            }
        }
    }
}

// ---- leaders, from the ranks: -1 leaves; a paired node's is the smaller of
// the pair; an unpaired node attached to a paired one joins that pair; of the
// others, two attached to each other pair up, one attached to a node that is
// itself not attached to an open node joins it, the rest lead themselves.

__device__ __forceinline__ int mate_of(const BuildArgs &a, const int32_t *best, int i) {
    const int p = a.partner[i];
    if (p != -1) return p;
    const int b = best[i];
    return b >= 0 && best[b] == i ? b : -1;
}

__device__ __forceinline__ int lead_first(const BuildArgs &a, const int32_t *best, int i) {
    const int p = mate_of(a, best, i);
    if (p == -3) return -1;
    if (p >= 0) return min(i, p);
    const int t = a.att[i];
    if (t >= 0) {
        const int q = mate_of(a, best, t);
        if (q >= 0) return min(t, q);
    }
    return -2;
}

__device__ __forceinline__ int wanted(const BuildArgs &a, const int32_t *best, int i) {  // i is open
    const int t = a.att[i];
    return t >= 0 && lead_first(a, best, t) == -2 ? t : -1;
}

__device__ __forceinline__ int leader_of(const BuildArgs &a, const int32_t *best, int i) {
    const int l = lead_first(a, best, i);
    if (l != -2) return l;
    const int t = wanted(a, best, i);
    if (t < 0) return i;
    const int b = wanted(a, best, t);
    if (b == i) return min(i, t);
    return b < 0 ? t : i;
}

// ---- coarse rows

__device__ __forceinline__ int pow2_at_least(int n) {
    int p = 32;
    while (p < n) p <<= 1;
    return p;
}

// Sorts keys[0, P) ascending with nt threads (tid in [0, nt)); sync() orders them.
template <class Sync> __device__ void bitonic(unsigned long long *keys, int P, int tid, int nt, Sync sync) {
    for (int k = 2; k <= P; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < P; i += nt) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long x = keys[i], y = keys[l];
                    if ((x > y) == ((i & k) == 0)) {
                        keys[i] = y;
                        keys[l] = x;
                    }
                }
            }
            sync();
        }
}

// Merges the sorted entries (key: coarse node << 32 | arrival; all ones: none)
// into the coarse row I, summing equal nodes in arrival order; one warp.
__device__ void merge_row(const HierView &v, int64_t noff2, int I, const unsigned long long *keys, const double *vals,
                          int n, int &len) {
    const int lane = threadIdx.x & 31;
    const int64_t dst = v.rs[noff2 + I];
    int runs = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const unsigned long long k = i < n ? keys[i] : ~0ull;
        const int J = static_cast<int>(k >> 32);
        const bool start = k != ~0ull && (i == 0 || static_cast<int>(keys[i - 1] >> 32) != J);
        const unsigned mask = __ballot_sync(0xffffffffu, start);
        if (start) {
            double s = vals[k & 0xffffffffull];
            for (int q = i + 1; q < n && static_cast<int>(keys[q] >> 32) == J && keys[q] != ~0ull; ++q)
                s += vals[keys[q] & 0xffffffffull];
            const int64_t at = dst + runs + __popc(mask & ((1u << lane) - 1u));
            v.ecol[at] = J;
            v.ew[at] = s;
        }
        runs += __popc(mask);
    }
    if (lane == 0) v.rl[noff2 + I] = runs;
    len = runs;
}

// Puts the cnt members at own[0, cnt) in node order (one warp).
__device__ void sort_members(int32_t *own, int cnt) {
    const int lane = threadIdx.x & 31;
    if (cnt <= 32) {
        const int m = lane < cnt ? own[lane] : 0x7fffffff;
        int rank = 0;
        for (int q = 0; q < cnt; ++q) rank += __shfl_sync(0xffffffffu, m, q) < m ? 1 : 0;
        __syncwarp();
        if (lane < cnt) own[rank] = m;
    } else if (lane == 0) {
        for (int p = 1; p < cnt; ++p) {
            const int m = own[p];
            int q = p;
            for (; q > 0 && own[q - 1] > m; --q) own[q] = own[q - 1];
            own[q] = m;
        }
    }
    __syncwarp();
}

// Coarse row I (raw <= kWarpRaw entries over its members), by one warp.
__device__ int coarse_row_warp(const BuildArgs &a, int64_t noff, int64_t noff2, int I, int raw, unsigned long long *keys,
                               double *vals) {
    const HierView &v = a.v;
    const int lane = threadIdx.x & 31;
    const int cnt = v.gc[noff2 + I];
    int32_t *own = v.own + noff + v.gs[noff2 + I];
    sort_members(own, cnt);
    double shift = 0.0;  // edges to nodes without coarse counterpart join the coarse excess
    int done = 0;        // entries of the members before this batch of 32
    for (int m0 = 0; m0 < cnt; m0 += 32) {
        const int m = m0 + lane < cnt ? own[m0 + lane] : -1;
        const int len = m >= 0 ? v.rl[noff + m] : 0;
        const int64_t e0 = m >= 0 ? v.rs[noff + m] : 0;
        int incl = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        const int nm = min(32, cnt - m0);
        for (int base = 0; base < tot; base += 32) {
            const int t = base + lane;
            int k = 0;  // the member holding raw entry t
            for (int q = 0; q < nm - 1; ++q) k += t >= __shfl_sync(0xffffffffu, incl, q) ? 1 : 0;
            const int before = __shfl_sync(0xffffffffu, incl - len, k);
            const int64_t e = __shfl_sync(0xffffffffu, e0, k) + (t - before);
            if (t < tot) {
                const int J = v.agg[noff + v.ecol[e]];
                const double w = v.ew[e];
                if (J < 0) shift += w;
                keys[done + t] = (J < 0 || J == I) ? ~0ull
                                                   : (static_cast<unsigned long long>(static_cast<unsigned>(J)) << 32) |
                                                         static_cast<unsigned>(done + t);
                vals[done + t] = w;
            }
        }
        done += tot;
    }
    if (__any_sync(0xffffffffu, shift != 0.0)) shift = warp_sum(shift);
    if (lane == 0) v.ex[noff2 + I] = shift;
    const int P = pow2_at_least(raw);
    for (int i = raw + lane; i < P; i += 32) keys[i] = ~0ull;
    __syncwarp();
    bitonic(keys, P, lane, 32, [] { __syncwarp(); });
    int len;
    merge_row(v, noff2, I, keys, vals, raw, len);
    __syncwarp();
    return len;
}

// A wider coarse row (raw <= kBlockRaw), by the whole block.
__device__ int coarse_row_block(const BuildArgs &a, int64_t noff, int64_t noff2, int I, int raw,
                                unsigned long long *keys, double *vals) {
    const HierView &v = a.v;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (wid == 0) {
        const int cnt = v.gc[noff2 + I];
        int32_t *own = v.own + noff + v.gs[noff2 + I];
        sort_members(own, cnt);
        double shift = 0.0;
        int done = 0;
        for (int k = 0; k < cnt; ++k) {
            const int m = own[k];
            const int len = v.rl[noff + m];
            const int64_t e0 = v.rs[noff + m];
            for (int e = lane; e < len; e += 32) {
                const int J = v.agg[noff + v.ecol[e0 + e]];
                const double w = v.ew[e0 + e];
                if (J < 0) shift += w;
                keys[done + e] = (J < 0 || J == I) ? ~0ull
                                                   : (static_cast<unsigned long long>(static_cast<unsigned>(J)) << 32) |
                                                         static_cast<unsigned>(done + e);
                vals[done + e] = w;
            }
            done += len;
        }
        shift = warp_sum(shift);
        if (lane == 0) v.ex[noff2 + I] = shift;
    }
    const int P = pow2_at_least(raw);
    for (int i = raw + threadIdx.x; i < P; i += blockDim.x) keys[i] = ~0ull;
    __syncthreads();
    bitonic(keys, P, threadIdx.x, blockDim.x, [] { __syncthreads(); });
    int len = 0;
    if (wid == 0) merge_row(v, noff2, I, keys, vals, raw, len);
    __syncthreads();
    return len;  // valid in warp 0
}

// The coarse rows g0 .. g1 - 1, one warp each, the wide ones by the whole block;
// then their diagonals.  Returns each warp's entries.
__device__ int coarse_rows(const BuildArgs &a, int64_t noff, int64_t noff2, int g0, int g1, unsigned long long *keys,
                           double *vals, int *s_count, int *s_wide) {
    const HierView &v = a.v;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int got = 0;
    for (int base = g0; base < g1; base += kBuildThreads) {
        const int cnt_here = min(kBuildThreads, g1 - base);
        __syncthreads();
        if (tid == 0) *s_count = 0;
        __syncthreads();
        for (int q = wid; q < cnt_here; q += kBuildThreads / 32) {
            const int I = base + q;
            const int raw = v.raw[noff2 + I];
            if (raw <= kWarpRaw)
                got += coarse_row_warp(a, noff, noff2, I, raw, keys + wid * kWarpRaw, vals + wid * kWarpRaw);
            else if (lane == 0)
                s_wide[atomicAdd(s_count, 1)] = I;
        }
        __syncthreads();
        const int nwide = *s_count;
        for (int q = 0; q < nwide; ++q) {
            const int I = s_wide[q];
            const int raw = v.raw[noff2 + I];
            if (raw > kBlockRaw) {  // block-uniform
                if (tid == 0) {
                    v.rl[noff2 + I] = 0;
                    v.ex[noff2 + I] = 1.0;
                    atomicExch(&v.H->overflow, 1);
                }
                continue;
            }
            const int len = coarse_row_block(a, noff, noff2, I, raw, keys, vals);
            if (wid == 0) got += len;
        }
    }
    __syncthreads();
    for (int I = g0 + tid; I < g1; I += kBuildThreads) {
        double ex = v.ex[noff2 + I];
        const int64_t o = noff + v.gs[noff2 + I];
        for (int q = 0; q < v.gc[noff2 + I]; ++q) ex += v.ex[noff + v.own[o + q]];
        finish_row(v, noff2 + I, ex, &a.partner[I]);
    }
    return got;
}

// ---- the coarsest level's inverse
//
// Elimination without subtractions: with weights w and excess ex the pivot is
// d_k = ex_k + sum_{j > k} w_kj, and eliminating k adds f w_kj to w_ij and f ex_k
// to ex_i, f = w_ik / d_k -- sums of positive terms, so a shift of 1e-14 of the
// weights keeps its relative precision.  The same steps applied to the unit
// matrix give M, and inv = sum_k M_k M_k^T / d_k, again sums of positive terms
// (its lower triangle, with the division folded into one factor: a third of the
// FP64 instructions, 10 of the 25 us that 32 nodes took).
// Row i holds w_ij for j above the pivot and M_ij below it, one warp per row and
// one lane per column: only the rows below the pivot issue FP64 instructions.
__device__ void dense_inverse(const HierView &v, int64_t noff, int n, double *sm) {
    double(*w)[kDense + 1] = reinterpret_cast<double(*)[kDense + 1]>(sm);
    double *ex = &w[kDense][0], *dinv = ex + kDense;
    const int i = threadIdx.x >> 5, j = threadIdx.x & 31;  // kBuildThreads = kDense^2
    w[i][j] = 0.0;
    __syncthreads();
    if (i < n) {
        const int64_t e0 = v.rs[noff + i];
        const int len = v.rl[noff + i];
        for (int e = j; e < len; e += 32) w[i][v.ecol[e0 + e]] = v.ew[e0 + e];
        if (j == 0) ex[i] = v.ex[noff + i];
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (i == k) {
            const double s = warp_sum(j > k && j < n ? w[k][j] : 0.0);
            if (j == 0) dinv[k] = 1.0 / (ex[k] + s);
        }
        __syncthreads();
        if (i > k && i < n) {  // warp-uniform
            const double f = w[i][k] * dinv[k];
            __syncwarp();
            if (j == k)
                w[i][k] = f;
            else if (j < n && j != i)
                w[i][j] += f * w[k][j];
            else if (j == i)
                ex[i] += f * ex[k];
        }
        __syncthreads();
    }
    // N_kj = M_kj / d_k in the places above the diagonal, which are done with
    if (i < n && j < i) w[j][i] = w[i][j] * dinv[i];
    __syncthreads();
    if (i < n && j <= i) {
        double s = j == i ? dinv[i] : w[j][i];
        for (int k = i + 1; k < n; ++k) s += w[k][i] * w[j][k];
        v.H->inv[i * kDense + j] = s;
        v.H->inv[j * kDense + i] = s;
    }
}

// ---- the build

// ONE: the grid is one cluster.
template <int LPR, bool ONE> __global__ void __launch_bounds__(kBuildThreads, 1) k_amg_build(const __grid_constant__ BuildArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(smem);
    double *vals = reinterpret_cast<double *>(smem + sizeof(unsigned long long) * kBlockRaw);
    __shared__ int pre[2][kMaxCtas + 1];
    __shared__ int tmp[33];
    __shared__ int s_base[2];
    __shared__ unsigned long long s_ebase;
    __shared__ int s_wide[kBuildThreads];
    const HierView &v = a.v;
    Hier *H = v.H;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int nb = gridDim.x, b = blockIdx.x;
    GridBarT<ONE> bar(&H->bar[0], &a.ip.st->err, gridDim.x);
    if (__syncthreads_or(a.ip.st->stop | a.ip.st->err)) return;
    if (b == 0) {  // the control block's values, for this build (behind the weights' barrier) and the solves
        if (!a.same && tid < kMaxLevels) {
            H->mcur[tid] = 0;
            H->nnzacc[tid] = 0;
        }
        if (tid < kMaxCtas / kWideCluster) H->left[0][tid] = 0;
        if (tid == 0) {
            if (!a.same) H->overflow = 0;
            if (!a.same) H->ecur = static_cast<unsigned long long>(a.e0);
            H->bar[1] = 0;
            H->notier[0] = 0;
            H->general = 0;
        }
    }
    {
        int64_t r0, r1;
        ip_range(a.nc, b, nb, r0, r1);
        if (!ip_weights(a.ip, bar, r0, r1)) return;
    }
    if (!bar.sync()) return;

    int n = a.n0;
    int64_t noff = 0, nnz = a.e0;
    int block_nodes = 0;  // nodes of the levels built by block 0 alone
    {
        const int ch = (n + nb - 1) / nb;
        level0_values<LPR>(a, min(n, b * ch), min(n, (b + 1) * ch));
    }
    if (!bar.sync()) return;
    if (a.same) {  // values alone, one pass per level
        const int nlev = H->nlev;
        for (int l = 0; l + 1 < nlev; ++l) {
            const LevelInfo F = H->L[l], C = H->L[l + 1];
            if (nb > 1 && !F.grid) {
                if (b != 0) return;
                nb = 1;
                bar.nb = 1;
            }
            const int ch = (C.n + nb - 1) / nb;
            const int g0 = min(C.n, b * ch), g1 = min(C.n, g0 + ch);
            coarse_rows(a, F.noff, C.noff, g0, g1, keys, vals, &s_base[1], s_wide);
            if (!bar.sync()) return;
        }
        const LevelInfo Z = H->L[nlev - 1];
        if (b == 0 && H->dense) dense_inverse(v, Z.noff, Z.n, reinterpret_cast<double *>(smem));
        return;
    }
    int l = 0, sweeps = kLargeSweeps;
    for (;; ++l) {
        if (nb > 1 && nnz <= kBlockEntries && n <= kBlockNodes) {
            if (b != 0) return;  // block 0 finishes the hierarchy alone
            nb = 1;
            bar.nb = 1;
        }
        const int grid = nb > 1 ? 1 : 0;
        if (b == 0 && tid == 0) {
            H->L[l].noff = noff;
            H->L[l].n = n;
            H->L[l].nmem = 0;
            H->L[l].nnz = nnz;
            H->L[l].grid = grid;
        }
        if (!grid && l > 0) block_nodes += n;
        if (n <= kDense || l + 1 == kMaxLevels) break;
        const int ch = (n + nb - 1) / nb;
        const int i0 = min(n, b * ch), i1 = min(n, i0 + ch);
        rank_round<LPR>(a, noff, i0, i1, 0, nullptr, a.best0);
        if (!bar.sync()) return;
        int32_t *bp = a.best0, *bc = a.best1;
        for (int r = 1; r < kHandshakes; ++r) {
            rank_round<LPR>(a, noff, i0, i1, r, bp, bc);
            if (!bar.sync()) return;
            int32_t *t = bp;
            bp = bc;
            bc = t;
        }
        // leaders and, per block, their number and that of the leaving nodes
        int run = 0, lrun = 0;
        for (int base = i0; base < i1; base += kBuildThreads) {
            const int i = base + tid;
            int lead = -2, flags = 0;
            if (i < i1) {
                lead = leader_of(a, bp, i);
                flags = lead == i ? 1 : (lead == -1 ? 1 << 16 : 0);
            }
            int tot;
            const int at = block_scan(flags, tmp, tot);
            if (i < i1) {
                a.lead[i] = lead;
                a.pos[i] = lead == i ? run + (at & 0xffff) : lrun + (at >> 16);
            }
            run += tot & 0xffff;
            lrun += tot >> 16;
        }
        if (tid == 0) {
            H->ctasum[0][b] = run;
            H->ctasum[1][b] = lrun;
        }
        if (!bar.sync()) return;
        // their prefixes over the blocks
        if (wid < 2) {
            int carry = 0;
            for (int base = 0; base < nb; base += 32) {
                const int q = base + lane;
                const int x = q < nb ? *reinterpret_cast<volatile int *>(&H->ctasum[wid][q]) : 0;
                int incl = x;
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (q < nb) pre[wid][q] = carry + incl - x;
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) pre[wid][nb] = carry;
        }
        __syncthreads();
        const int nco = pre[0][nb], nlv = pre[1][nb], active = n - nlv;
        const int64_t noff2 = noff + n;
        if (active == 0) sweeps = kDominantSweeps;
        if (active == 0 || nco < 1 || nco >= active * kStall || noff2 + nco > v.capn ||
            (!grid && l > 0 && block_nodes + nco > kBlockTotalNodes))
            break;
        // aggregates: members are counted and their raw entries added up
        for (int i = i0 + tid; i < i1; i += kBuildThreads) {
            const int L = a.lead[i];
            int I = -1;
            if (L < 0) {
                v.own[noff + active + pre[1][b] + a.pos[i]] = i;
            } else {
                I = pre[0][L / ch] + a.pos[L];
                atomicAdd(&a.cnt[I], 1);
                atomicAdd(&a.cap[I], v.rl[noff + i]);
            }
            v.agg[noff + i] = I;
        }
        if (!bar.sync()) return;
        // per block of coarse nodes: where their members and entries go
        const int ch2 = (nco + nb - 1) / nb;
        const int g0 = min(nco, b * ch2), g1 = min(nco, g0 + ch2);
        int mtot = 0;
        int64_t etot = 0;
        for (int pass = 0; pass < 2; ++pass) {  // totals first, then the places
            int m = 0;
            int64_t e = 0;
            for (int base = g0; base < g1; base += kBuildThreads) {
                const int I = base + tid;
                const int c = I < g1 ? a.cnt[I] : 0, cp = I < g1 ? a.cap[I] : 0;
                int ct, et;
                const int ca = block_scan(c, tmp, ct);
                const int ea = block_scan(cp, tmp, et);
                if (pass == 1 && I < g1) {
                    v.gs[noff2 + I] = s_base[0] + m + ca;
                    v.gc[noff2 + I] = c;
                    v.raw[noff2 + I] = cp;
                    v.rs[noff2 + I] = static_cast<int64_t>(s_ebase) + e + ea;
                    a.cnt[I] = 0;  // from here on the members placed so far
                }
                m += ct;
                e += et;
            }
            if (pass == 0) {
                mtot = m;
                etot = e;
                __syncthreads();
                if (tid == 0) {
                    s_base[0] = static_cast<int>(atomicAdd(&H->mcur[l], static_cast<unsigned>(mtot)));
                    s_ebase = atomicAdd(&H->ecur, static_cast<unsigned long long>(etot));
                    if (s_ebase + etot > static_cast<unsigned long long>(v.cape)) atomicExch(&H->overflow, 1);
                    Seg s;
                    s.m0 = s_base[0];
                    s.mlen = mtot;
                    s.l0 = active + pre[1][b];
                    s.llen = pre[1][b + 1] - pre[1][b];
                    s.g0 = g0;
                    s.glen = g1 - g0;
                    v.seg[l * kMaxCtas + b] = s;
                }
                __syncthreads();
            }
        }
        if (!bar.sync()) return;
        if (*reinterpret_cast<volatile int *>(&H->overflow)) break;  // the finer level stays the coarsest
        for (int i = i0 + tid; i < i1; i += kBuildThreads) {
            const int I = v.agg[noff + i];
            if (I >= 0) v.own[noff + v.gs[noff2 + I] + atomicAdd(&a.cnt[I], 1)] = i;
        }
        if (!bar.sync()) return;
        const int got = coarse_rows(a, noff, noff2, g0, g1, keys, vals, &s_base[1], s_wide);
        if (lane == 0 && got) atomicAdd(&H->nnzacc[l + 1], static_cast<unsigned long long>(got));
        if (!bar.sync()) return;
        if (*reinterpret_cast<volatile int *>(&H->overflow)) break;
        if (b == 0 && tid == 0) H->L[l].nmem = active;
        nnz = static_cast<int64_t>(*reinterpret_cast<volatile unsigned long long *>(&H->nnzacc[l + 1]));
        n = nco;
        noff = noff2;
    }
    // level l is the coarsest
    if (b != 0) return;
    const int dense = n <= kDense ? 1 : 0;
    if (dense) dense_inverse(v, noff, n, reinterpret_cast<double *>(smem));
    if (tid == 0) {
        H->nlev = l + 1;
        H->dense = dense;
        H->sweeps = sweeps;
    }
}

// ---- host side

SolveShape solve_shape(bchar_mesh_t m) {
    Amg &A = m->amg;
    if (!A.resident) {
        const SolveRoom r = solve_room();
        A.resident = r.blocks;
        A.small_fits = r.small && build_cluster_fits();
    }
    return solve_shape_of(A.e0, A.n0, {A.resident, A.small_fits});
}

// All blocks resident at once: one cluster, or a cooperative launch.
template <typename... P, typename... A>
static void launch_resident(void (*kernel)(P...), int grid, bool cluster, int block, size_t smem, cudaStream_t s,
                            A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    if (cluster) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = grid;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

void amg_opt_in() {
    for (auto k : {k_amg_build<4, false>, k_amg_build<16, false>, k_amg_build<4, true>, k_amg_build<16, true>}) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBuildSmem));
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
}

bool build_cluster_fits() {
    int n = 0, least = 1 << 30;
    for (auto k : {k_amg_build<4, true>, k_amg_build<16, true>}) {
        if (!clusters_resident(k, kSmallCluster, kBuildThreads, kBuildSmem, &n)) return false;
        least = n < least ? n : least;
    }
    return least >= 1;
}

HierView hier_view(bchar_mesh_t m) {
    Amg &A = m->amg;
    HierView v{};
    v.H = ptr<Hier>(A.hier);
    v.seg = ptr<Seg>(A.seg);
    v.capn = A.capn;
    v.cape = A.cape;
    v.rs = ptr<int64_t>(A.rs);
    v.rl = ptr<int32_t>(A.rl);
    v.dg = ptr<double>(A.dg);
    v.ex = ptr<double>(A.ex);
    v.om = ptr<double>(A.om);
    v.x = ptr<double>(A.x);
    v.b = ptr<double>(A.b);
    v.own = ptr<int32_t>(A.own);
    v.gs = ptr<int32_t>(A.gs);
    v.gc = ptr<int32_t>(A.gc);
    v.agg = ptr<int32_t>(A.agg);
    v.raw = ptr<int32_t>(A.raw);
    v.ecol = ptr<int32_t>(A.ecol);
    v.ew = ptr<double>(A.ew);
    return v;
}

void amg_build(bchar_mesh_t m, const IpArgs &ip, bool same_aggregates) {
    Amg &A = m->amg;
    BuildArgs a{};
    a.v = hier_view(m);
    a.n0 = static_cast<int>(A.n0);
    a.e0 = A.e0;
    a.schur = A.schur ? 1 : 0;
    a.nc = m->nc;
    a.col_ptr = ptr<int64_t>(m->col_ptr);
    a.csc_row = ptr<int32_t>(m->csc_row);
    a.a2 = ptr<double>(m->a2);
    a.a2c = ptr<double>(m->a2c);
    a.diag = ptr<double>(m->diag);
    a.exc = ptr<double>(m->qexc);
    a.g = ptr<double>(A.g);
    a.t = ptr<double>(A.t);
    a.cs = ptr<uint32_t>(A.cs);
    a.pair = ptr<int2>(A.pair);
    int32_t *s = ptr<int32_t>(A.scratch);
    int32_t **dst[] = {&a.best0, &a.best1, &a.partner, &a.att, &a.lead, &a.pos, &a.cnt, &a.cap};
    for (int32_t **d : dst) {
        *d = s;
        s += A.n0;
    }
    a.ip = ip;
    a.same = same_aggregates ? 1 : 0;
    const SolveShape shape = solve_shape(m);
    const bool few = A.e0 <= 10 * A.n0;  // lanes per row
    launch_resident(shape.small ? (few ? k_amg_build<4, true> : k_amg_build<16, true>)
                                : (few ? k_amg_build<4, false> : k_amg_build<16, false>),
                    shape.grid, shape.small, kBuildThreads, kBuildSmem, m->stream, a);
    ++m->launches;
}

void amg_release(Amg &A) {
    Buf *all[] = {&A.hier, &A.seg, &A.rs, &A.rl, &A.dg, &A.ex, &A.om, &A.x, &A.b, &A.own, &A.gs, &A.gc, &A.agg, &A.raw, &A.ecol, &A.ew,
                  &A.g, &A.t, &A.cs, &A.pair, &A.scratch, &A.raw_cnt, &A.raw_off, &A.raw_key, &A.vec, &A.stat};
    for (Buf *b : all) release(*b);
}

}  // namespace bchar
