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
    int32_t *best0, *best1, *partner, *att, *lead, *pos, *agg, *cnt, *cap;  // n0 each
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
__device__ __forceinline__ unsigned long long edge_rank(int i, int j, double w) {
    const unsigned long long cls = (static_cast<unsigned long long>(__double_as_longlong(w)) >> 52) & 0x7ffull;
    return (cls << 32) | edge_hash(i, j);
}

// The higher-ranked of (key, j) and (k2, j2); j < 0 is none; ties go to the smaller node.
__device__ __forceinline__ void take_higher(unsigned long long &key, int &j, unsigned long long k2, int j2) {
    if (j2 >= 0 && (j < 0 || k2 > key || (k2 == key && j2 < j))) {
        key = k2;
        j = j2;
    }
}

__device__ __forceinline__ bool leaves(const HierView &v, int64_t k) {
    return v.rl[k] == 0 || v.ex[k] >= (1.0 - kDominant) * v.dg[k];
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

// ---- the finest level's values: LPR lanes per row

template <int LPR> __device__ void level0_values(const BuildArgs &a, int i0, int i1) {
    const int lane = threadIdx.x & 31, sub = lane % LPR;
    const HierView &v = a.v;
    for (int r0 = i0 + static_cast<int>(threadIdx.x >> 5) * (32 / LPR); r0 < i1; r0 += blockDim.x / LPR) {
        const int i = r0 + lane / LPR;
        const bool ok = i < i1;
        double s = 0.0, x = 0.0;
        int len = 0;
        if (ok) {
            const int64_t e0 = v.rs[i];
            len = v.rl[i];
            if (a.schur) {
                for (int e = sub; e < len; e += LPR) {
                    double w = 0.0;
                    const uint32_t k1 = a.cs[e0 + e + 1];
                    for (uint32_t k = a.cs[e0 + e]; k < k1; ++k) {
                        const int2 p = a.pair[k];
                        w += a.g[p.x] * a.g[p.y];
                    }
                    v.ew[e0 + e] = w;
                    s += w;
                }
                for (int64_t p = a.col_ptr[i] + sub; p < a.col_ptr[i + 1]; p += LPR) x += a.a2c[p] * a.t[a.csc_row[p]];
            } else {
                const bool row = i < a.nc;
                const int64_t src = row ? e0 : a.col_ptr[i - a.nc];  // the row entries come first, in CSR order
                for (int e = sub; e < len; e += LPR) v.ew[e0 + e] = row ? a.a2[src + e] : a.a2c[src + e];
            }
        }
        for (int o = LPR / 2; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            x += __shfl_xor_sync(0xffffffffu, x, o);
        }
        if (ok && sub == 0) {
            const double ex = a.schur ? a.exc[a.nc + i] + x : a.exc[i];
            const double d = a.schur ? ex + s : a.diag[i];
            v.ex[i] = ex;
            v.dg[i] = d;
            v.om[i] = (len == 0 ? 1.0 : kOmega) / d;
        }
    }
}

// ---- one matching round (LPR lanes per node of the level at node offset noff)

template <int LPR>
__device__ void rank_round(const BuildArgs &a, int64_t noff, int n, int i0, int i1, int round, const int32_t *bprev,
                           int32_t *bcur) {
    const HierView &v = a.v;
    const int lane = threadIdx.x & 31, sub = lane % LPR;
    volatile int32_t *partner = a.partner;
    for (int r0 = i0 + static_cast<int>(threadIdx.x >> 5) * (32 / LPR); r0 < i1; r0 += blockDim.x / LPR) {
        const int i = r0 + lane / LPR;
        const bool ok = i < i1;
        unsigned long long key = 0, akey = 0;
        int bj = -1, aj = -1, mate = -3;
        double wmax = 0.0, di = 0.0;
        if (ok) {
            di = v.dg[noff + i];
            if (round == 0) {
                mate = leaves(v, noff + i) ? -3 : -1;
            } else {
                mate = partner[i];
                if (mate == -1) {  // did the previous round's choices meet?
                    const int b = bprev[i];
                    if (b >= 0 && bprev[b] == i) mate = b;
                }
            }
            const bool open = mate == -1;
            if (open) {
                const int64_t e0 = v.rs[noff + i];
                const int len = v.rl[noff + i];
                for (int e = sub; e < len; e += LPR) {
                    const int j = v.ecol[e0 + e];
                    const double w = v.ew[e0 + e];
                    if (!(w > 0.0)) continue;
                    if (round == 0) {
                        if (leaves(v, noff + j)) continue;
                    } else {
                        if (partner[j] != -1) continue;
                        const int b = bprev[j];
                        if (b >= 0 && bprev[b] == j) continue;
                    }
                    const unsigned long long k = edge_rank(i, j, w);
                    if (round == 0) {
                        wmax = fmax(wmax, w);
                        take_higher(akey, aj, k, j);
                    }
                    // strong: w >= kStrength sqrt(d_i d_j), compared squared
                    if (w * w >= (kStrength * kStrength) * (di * v.dg[noff + j])) take_higher(key, bj, k, j);
                }
            }
        }
        for (int o = LPR / 2; o > 0; o >>= 1) {
            take_higher(key, bj, __shfl_xor_sync(0xffffffffu, key, o), __shfl_xor_sync(0xffffffffu, bj, o));
            if (round == 0) {
                take_higher(akey, aj, __shfl_xor_sync(0xffffffffu, akey, o), __shfl_xor_sync(0xffffffffu, aj, o));
                wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
            }
        }
        if (ok && sub == 0) {
            bcur[i] = bj;
            partner[i] = mate;
            if (round == 0) {
                // one-sided on purpose: a leaf hanging off a hub by an edge that is most of
                // its own diagonal but little of the hub's should follow the hub
                a.att[i] = (aj >= 0 && wmax >= kAttach * di) ? aj : -1;
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
                          int n, double ex, int &len) {
    const int lane = threadIdx.x & 31;
    const int64_t dst = v.rs[noff2 + I];
    int runs = 0;
    double d = 0.0;
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
            d += s;
        }
        runs += __popc(mask);
    }
    d = warp_sum(d) + ex;
    if (lane == 0) {
        v.rl[noff2 + I] = runs;
        v.dg[noff2 + I] = d;
        v.ex[noff2 + I] = ex;
        v.om[noff2 + I] = (runs == 0 ? 1.0 : kOmega) / d;
    }
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
    double ex = 0.0;
    int done = 0;  // entries of the members before this batch of 32
    for (int m0 = 0; m0 < cnt; m0 += 32) {
        const int m = m0 + lane < cnt ? own[m0 + lane] : -1;
        const int len = m >= 0 ? v.rl[noff + m] : 0;
        const int64_t e0 = m >= 0 ? v.rs[noff + m] : 0;
        if (m >= 0) ex += v.ex[noff + m];
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
                const int J = a.agg[v.ecol[e]];
                const double w = v.ew[e];
                if (J < 0) ex += w;  // an edge to a node without coarse counterpart joins the shift
                keys[done + t] = (J < 0 || J == I) ? ~0ull
                                                   : (static_cast<unsigned long long>(static_cast<unsigned>(J)) << 32) |
                                                         static_cast<unsigned>(done + t);
                vals[done + t] = w;
            }
        }
        done += tot;
    }
    ex = warp_sum(ex);
    const int P = pow2_at_least(raw);
    for (int i = raw + lane; i < P; i += 32) keys[i] = ~0ull;
    __syncwarp();
    bitonic(keys, P, lane, 32, [] { __syncwarp(); });
    int len;
    merge_row(v, noff2, I, keys, vals, raw, ex, len);
    __syncwarp();
    return len;
}

// A wider coarse row (raw <= kBlockRaw), by the whole block.
__device__ int coarse_row_block(const BuildArgs &a, int64_t noff, int64_t noff2, int I, int raw,
                                unsigned long long *keys, double *vals, double *ex_sm) {
    const HierView &v = a.v;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (wid == 0) {
        const int cnt = v.gc[noff2 + I];
        int32_t *own = v.own + noff + v.gs[noff2 + I];
        sort_members(own, cnt);
        double ex = 0.0;
        int done = 0;
        for (int k = 0; k < cnt; ++k) {
            const int m = own[k];
            const int len = v.rl[noff + m];
            const int64_t e0 = v.rs[noff + m];
            if (lane == 0) ex += v.ex[noff + m];
            for (int e = lane; e < len; e += 32) {
                const int J = a.agg[v.ecol[e0 + e]];
                const double w = v.ew[e0 + e];
                if (J < 0) ex += w;
                keys[done + e] = (J < 0 || J == I) ? ~0ull
                                                   : (static_cast<unsigned long long>(static_cast<unsigned>(J)) << 32) |
                                                         static_cast<unsigned>(done + e);
                vals[done + e] = w;
            }
            done += len;
        }
        ex = warp_sum(ex);
        if (lane == 0) *ex_sm = ex;
    }
    const int P = pow2_at_least(raw);
    for (int i = raw + threadIdx.x; i < P; i += blockDim.x) keys[i] = ~0ull;
    __syncthreads();
    bitonic(keys, P, threadIdx.x, blockDim.x, [] { __syncthreads(); });
    int len = 0;
    if (wid == 0) merge_row(v, noff2, I, keys, vals, raw, *ex_sm, len);
    __syncthreads();
    return len;  // valid in warp 0
}

// ---- the coarsest level's inverse
//
// Elimination without subtractions: with weights w and excess ex the pivot is
// ex_k + sum_{j > k} w_kj, and eliminating k adds w_ik w_kj / d_k to w_ij and
// w_ik ex_k / d_k to ex_i -- sums of positive terms, so a shift of 1e-14 of the
// weights keeps its relative precision.  L = (I - F) with F >= 0 gives
// inv = sum_k M_k M_k^T / d_k, M = (I - F)^{-1}, again sums of positive terms.
__device__ void dense_inverse(const HierView &v, int64_t noff, int n, double *sm) {
    double(*w)[kDense + 1] = reinterpret_cast<double(*)[kDense + 1]>(sm);
    double(*M)[kDense + 1] = w + kDense;
    double *ex = &M[kDense][0], *d = ex + kDense;
    const int i = threadIdx.x >> 5, j = threadIdx.x & 31;  // kBuildThreads = kDense^2
    w[i][j] = 0.0;
    M[i][j] = 0.0;
    __syncthreads();
    if (i < n) {
        const int64_t e0 = v.rs[noff + i];
        const int len = v.rl[noff + i];
        for (int e = j; e < len; e += 32) w[i][v.ecol[e0 + e]] = v.ew[e0 + e];
        if (j == 0) ex[i] = v.ex[noff + i];
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (i == 0) {
            double s = j > k && j < n ? w[k][j] : 0.0;
            s = warp_sum(s);
            if (j == 0) d[k] = ex[k] + s;
        }
        __syncthreads();
        const double dk = d[k], wik = w[i][k], wkj = w[k][j], exk = ex[k];
        __syncthreads();
        if (i > k && i < n) {
            const double f = wik / dk;
            if (j > k && j < n && j != i) w[i][j] += f * wkj;
            if (j == k) {
                ex[i] += f * exk;
                w[i][k] = f;  // F below the diagonal
            }
        }
        __syncthreads();
    }
    if (i == 0)  // column j of M, by lane j
        for (int r = 0; r < n; ++r) {
            double s = r == j ? 1.0 : 0.0;
            for (int k = j; k < r; ++k) s += w[r][k] * M[k][j];
            if (j < n) M[r][j] = r >= j ? s : 0.0;
        }
    __syncthreads();
    if (i < n && j < n) {
        double s = 0.0;
        for (int k = max(i, j); k < n; ++k) s += M[k][i] * M[k][j] / d[k];
        v.H->inv[i * kDense + j] = s;
    }
}

// ---- the build

template <int LPR> __global__ void __launch_bounds__(kBuildThreads, 1) k_amg_build(BuildArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(smem);
    double *vals = reinterpret_cast<double *>(smem + sizeof(unsigned long long) * kBlockRaw);
    __shared__ int pre[2][kMaxCtas + 1];
    __shared__ int tmp[33];
    __shared__ int s_base[2];
    __shared__ unsigned long long s_ebase;
    __shared__ double s_ex;
    __shared__ int s_wide[kBuildThreads];
    const HierView &v = a.v;
    Hier *H = v.H;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int nb = gridDim.x, b = blockIdx.x;
    GridBar bar(&H->bar[0], &H->err, gridDim.x);

    int n = a.n0;
    int64_t noff = 0, nnz = a.e0;
    int block_nodes = 0;  // nodes of the levels built by block 0 alone
    {
        const int ch = (n + nb - 1) / nb;
        level0_values<LPR>(a, min(n, b * ch), min(n, (b + 1) * ch));
        if (b == 0 && tid == 0) H->ecur = static_cast<unsigned long long>(a.e0);
    }
    if (!bar.sync()) return;
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
            H->L[l].grid = l == 0 ? 1 : grid;
        }
        if (!grid && l > 0) block_nodes += n;
        if (n <= kDense || l + 1 == kMaxLevels) break;
        const int ch = (n + nb - 1) / nb;
        const int i0 = min(n, b * ch), i1 = min(n, i0 + ch);
        rank_round<LPR>(a, noff, n, i0, i1, 0, nullptr, a.best0);
        if (!bar.sync()) return;
        int32_t *bp = a.best0, *bc = a.best1;
        for (int r = 1; r < kHandshakes; ++r) {
            rank_round<LPR>(a, noff, n, i0, i1, r, bp, bc);
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
            a.agg[i] = I;
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
            const int I = a.agg[i];
            if (I >= 0) v.own[noff + v.gs[noff2 + I] + atomicAdd(&a.cnt[I], 1)] = i;
        }
        if (!bar.sync()) return;
        // coarse rows: one warp each, the wide ones by the whole block
        int got = 0, nwide = 0;
        for (int base = g0; base < g1; base += kBuildThreads) {
            const int cnt_here = min(kBuildThreads, g1 - base);
            __syncthreads();
            if (tid == 0) s_base[1] = 0;
            __syncthreads();
            for (int q = wid; q < cnt_here; q += kBuildThreads / 32) {
                const int I = base + q;
                const int raw = a.cap[I];
                if (raw <= kWarpRaw)
                    got += coarse_row_warp(a, noff, noff2, I, raw, keys + wid * kWarpRaw, vals + wid * kWarpRaw);
                else if (lane == 0)
                    s_wide[atomicAdd(&s_base[1], 1)] = I;
            }
            __syncthreads();
            nwide = s_base[1];
            for (int q = 0; q < nwide; ++q) {
                const int I = s_wide[q];
                const int raw = a.cap[I];
                if (raw > kBlockRaw) {  // block-uniform
                    if (tid == 0) {
                        v.rl[noff2 + I] = 0;
                        v.dg[noff2 + I] = v.ex[noff2 + I] = v.om[noff2 + I] = 1.0;
                        atomicExch(&H->overflow, 1);
                    }
                    continue;
                }
                const int len = coarse_row_block(a, noff, noff2, I, raw, keys, vals, &s_ex);
                if (wid == 0) got += len;
            }
        }
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
        if (l > 0 && nb > 1) H->L[l].grid = 1;
    }
}

// ---- host side

int solve_grid(int64_t e0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    if (sms > kMaxCtas) sms = kMaxCtas;
    // one block per ~800 entries: the FP64 pipe takes about 1.7 products per
    // clock and SM, so a pass then costs ~500 clocks against ~2 300 for the barrier
    // after it; up to one block's worth of work needs no grid barrier at all
    int64_t g = e0 / 800;
    if (e0 <= 6000) g = 1;
    return static_cast<int>(g < 1 ? 1 : (g > sms ? sms : g));
}

template <typename... P, typename... A>
static void launch_cooperative(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
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
    v.ecol = ptr<int32_t>(A.ecol);
    v.ew = ptr<double>(A.ew);
    return v;
}

void amg_build(bchar_mesh_t m) {
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
    int32_t **dst[] = {&a.best0, &a.best1, &a.partner, &a.att, &a.lead, &a.pos, &a.agg, &a.cnt, &a.cap};
    for (int32_t **d : dst) {
        *d = s;
        s += A.n0;
    }
    cudaMemsetAsync(A.hier.p, 0, offsetof(Hier, L), m->stream);
    static bool attrs = false;  // the shared-memory opt-in (harmless to repeat)
    if (!attrs) {
        cudaFuncSetAttribute(k_amg_build<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBuildSmem));
        cudaFuncSetAttribute(k_amg_build<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBuildSmem));
        attrs = true;
    }
    const int grid = solve_grid(A.e0);
    if (A.e0 <= 10 * A.n0)
        launch_cooperative(k_amg_build<4>, grid, kBuildThreads, kBuildSmem, m->stream, a);
    else
        launch_cooperative(k_amg_build<16>, grid, kBuildThreads, kBuildSmem, m->stream, a);
    ++m->launches;
}

void amg_release(Amg &A) {
    Buf *all[] = {&A.hier, &A.seg, &A.rs, &A.rl, &A.dg, &A.ex, &A.om, &A.x, &A.b, &A.own, &A.gs, &A.gc, &A.ecol, &A.ew,
                  &A.g, &A.t, &A.cs, &A.pair, &A.scratch, &A.raw_cnt, &A.raw_off, &A.raw_key, &A.vec, &A.stat};
    for (Buf *b : all) release(*b);
}

}  // namespace bchar
