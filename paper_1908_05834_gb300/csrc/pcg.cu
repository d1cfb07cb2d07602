// Preconditioned conjugate gradients on the normal equations of the
// minimisation, one cooperative kernel per solve.
//
// Each iteration is a product with the finest level, a vector update and one
// V-cycle (a damped-Jacobi sweep before and after the coarse correction, the
// coarsest level solved by its inverse): two dependent passes per level and
// three more.  Launched pass by pass they cost 2.5 us each whatever their size,
// plus one block cycling every level of up to 4 096 nodes through global memory
// with 40 sweeps at the bottom: 0.13 ms per iteration at 32^2, 0.22 ms at
// 128^2, 0.35 ms at 24^3, for 5 to 30 us of arithmetic and memory traffic.
// Here the whole solve is one launch, with a grid barrier (1.2 us) between the
// passes of the large levels.  What bounds it is that latency on meshes up to
// ~10^5 cells and the FP64 pipe (about 1.7 products per clock and SM) beyond:
//   - restriction is fused with the residual and the next level's first sweep:
//     the group of threads of a coarse node sums the residual over its members'
//     rows, so a level takes one pass down; prolongation is fused with the sweep
//     of the level above: one pass up;
//   - a block owns the rows of its aggregates' members for the whole solve and
//     keeps them (columns, weights, diagonals) in shared memory as far as they
//     fit, finest level first, so a pass gathers the vector from L2 and nothing else;
//   - the direction p = z + beta p is formed by the readers of p (two gathers
//     instead of a pass of its own) unless the level is so large that the extra
//     FP64 work outweighs a barrier (kFuseEntries);
//   - levels of at most kBlockEntries entries are cycled by block 0 alone, rows
//     and vectors in its shared memory, between block barriers;
//   - the stopping test runs on the device in every block (the same fixed-order
//     sums everywhere), so a solve ends exactly when it has converged.
#include "amg.cuh"
#include "device.cuh"
#include "gridbar.cuh"

namespace bchar {

constexpr int kNT = kSolveThreads;
constexpr size_t kSolveSmem = 200 * 1024;  // dynamic shared memory: the cached rows
// entries per block of the grid beyond which p is formed by its own pass
constexpr int64_t kFuseEntries = 5000;

struct PcgArgs {
    HierView v;
    int n0;
    int64_t e0;
    int schur;
    int64_t nc;
    const int64_t *row_ptr, *col_ptr;
    const int32_t *col, *csc_row;
    const double *a2, *a2c, *diag, *rhs;  // the system on rows and columns
    double *dy;                           // its solution
    double *d, *r, *p0, *p1, *q, *z;      // finest level
    const double *b_row, *volphi;
    const double *scal;  // mu, rp_max
    SolveTol tol;
    int which;    // 0: from zero, 1: from d
    int vcycle;   // 1: one V-cycle only (timing)
    SolveStat *st;
};

// A block's share of a level shared by all blocks.
struct Share {
    int64_t noff;
    int n, nrow, mlen, ngrp, g0, first, lfirst;
    int lpr, lprg;
    int whole;   // 1: the rows are first .. first + nrow - 1 themselves (a coarsest level)
    int cached;
    const int *id, *off, *col, *gst;
    const double *w, *dg, *om;
};

// A level cycled by block 0 alone.
struct Tier {
    int64_t noff;
    int n, ng, lpr, lprg, cached;
    int *off, *own, *gs;
    const int *col;
    const double *w;
    double *dg, *om, *x, *b;
};

struct Row {
    int id, len;
    const int *col;
    const double *w;
    double dg, om;
};

__device__ __forceinline__ Row share_row(const HierView &v, const Share &S, int k) {
    Row r;
    if (S.cached) {
        const int o = S.off[k];
        r.id = S.id[k];
        r.len = S.off[k + 1] - o;
        r.col = S.col + o;
        r.w = S.w + o;
        r.dg = S.dg[k];
        r.om = S.om[k];
    } else {
        r.id = S.whole ? S.first + k : v.own[S.noff + (k < S.mlen ? S.first + k : S.lfirst + k - S.mlen)];
        const int64_t e = v.rs[S.noff + r.id];
        r.len = v.rl[S.noff + r.id];
        r.col = v.ecol + e;
        r.w = v.ew + e;
        r.dg = v.dg[S.noff + r.id];
        r.om = v.om[S.noff + r.id];
    }
    return r;
}

__device__ __forceinline__ Row tier_row(const HierView &v, const Tier &T, int i) {
    Row r;
    const int o = T.off[i];
    r.id = i;
    r.len = T.off[i + 1] - o;
    if (T.cached) {
        r.col = T.col + o;
        r.w = T.w + o;
    } else {
        const int64_t e = v.rs[T.noff + i];
        r.col = v.ecol + e;
        r.w = v.ew + e;
    }
    r.dg = T.dg[i];
    r.om = T.om[i];
    return r;
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
    for (; e + LPR < r.len; e += 2 * LPR) {
        const double x0 = x[r.col[e]], x1 = x[r.col[e + LPR]];
        s += r.w[e] * x0;
        s += r.w[e + LPR] * x1;
    }
    if (e < r.len) s += r.w[e] * x[r.col[e]];
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

#define WITH_LANES(L, CALL)                             \
    switch (L) {                                        \
    case 1: { constexpr int LPR = 1; CALL; } break;     \
    case 2: { constexpr int LPR = 2; CALL; } break;     \
    case 4: { constexpr int LPR = 4; CALL; } break;     \
    case 8: { constexpr int LPR = 8; CALL; } break;     \
    default: { constexpr int LPR = 16; CALL; } break;   \
    }

// Lanes per item: as many as keep the block's threads busy, but at least two
// entries each (every doubling adds one FP64 addition per lane to the sum).
__device__ __forceinline__ int lanes_for_items(int items, double mean) {
    int l = 1;
    while (l < 16 && 4 * l <= mean && items * 2 * l <= kNT) l *= 2;
    return l;
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

struct Shared {
    Share lev[kMaxLevels];
    Tier tier[kMaxLevels];
    double red[3][kNT];
    double red4[3][4];
    double out[3];
    int tmp[33];
    int nlev, ng, dense, sweeps;
    double *alt;  // second vector of a coarsest level swept by block 0
    double *inv;
};

__device__ __forceinline__ unsigned char *take(unsigned char *&p, size_t bytes) {
    unsigned char *q = p;
    p += (bytes + 15) & ~static_cast<size_t>(15);
    return q;
}

// Sums (slots 0, 1) and maximum (slot 2) of the threads' values, thread 0 of
// the block gets them in out; four warps per slot, fixed order.
__device__ __forceinline__ void block_partials(Shared &sh, int slots, double a, double b, double mx) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    sh.red[0][tid] = a;
    if (slots > 1) {
        sh.red[1][tid] = b;
        sh.red[2][tid] = mx;
    }
    __syncthreads();
    const int slot = wid >> 2;
    if (slot < slots) {
        const double *v = sh.red[slot] + (wid & 3) * (kNT / 4);
        double s = v[lane];
        for (int q = 32 + lane; q < kNT / 4; q += 32) s = slot == 2 ? fmax(s, v[q]) : s + v[q];
        for (int o = 16; o > 0; o >>= 1) {
            const double t = __shfl_xor_sync(0xffffffffu, s, o);
            s = slot == 2 ? fmax(s, t) : s + t;
        }
        if (lane == 0) sh.red4[slot][wid & 3] = s;
    }
    __syncthreads();
    if (tid < slots) {
        const double *f = sh.red4[tid];
        sh.out[tid] = tid == 2 ? fmax(fmax(f[0], f[1]), fmax(f[2], f[3])) : (f[0] + f[1]) + (f[2] + f[3]);
    }
    __syncthreads();
}

// The same over the blocks' partials at part[slot0 ..], result in out for every thread.
__device__ __forceinline__ void grid_totals(Shared &sh, const Hier *H, int slot0, int slots, unsigned nb) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < slots) {
        const volatile double *v = H->part[slot0 + wid];
        double s = 0.0;
        for (unsigned q = lane; q < nb; q += 32) s = wid == 2 ? fmax(s, v[q]) : s + v[q];
        for (int o = 16; o > 0; o >>= 1) {
            const double t = __shfl_xor_sync(0xffffffffu, s, o);
            s = wid == 2 ? fmax(s, t) : s + t;
        }
        if (lane == 0) sh.out[wid] = s;
    }
    __syncthreads();
}

// ---- the passes of a level shared by all blocks

// b and x of the next level: the residual b - L x summed over each aggregate,
// and that level's first sweep from zero.
template <int LPR>
__device__ void pass_down(const HierView &v, const Share &S, const double *bl, const double *x, int64_t noff2,
                          double *bc, double *xc) {
    for_items<LPR>(S.ngrp, [&](bool ok, int sub, int g) {
        double s = 0.0;
        if (ok) {
            int k0, k1;
            if (S.cached) {
                k0 = S.gst[g];
                k1 = S.gst[g + 1];
            } else {
                k0 = v.gs[noff2 + S.g0 + g] - S.first;
                k1 = k0 + v.gc[noff2 + S.g0 + g];
            }
            for (int k = k0; k < k1; ++k) {
                const Row r = share_row(v, S, k);
                if (sub == 0) s += bl[r.id] - r.dg * x[r.id];
                s += lane_dot<LPR>(r, sub, x);
            }
        }
        s = lanes_sum<LPR>(s);
        if (ok && sub == 0) {
            const int I = S.g0 + g;
            bc[I] = s;
            xc[I] = v.om[noff2 + I] * s;
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
template <int LPR>
__device__ void pass_up(const HierView &v, const Share &S, const double *bl, const double *x, int64_t fine, double *xf) {
    for_items<LPR>(S.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        double xi = 0.0, bi = 0.0;
        if (ok) {
            r = share_row(v, S, k);
            xi = x[r.id];
            bi = bl[r.id];
            s = lane_dot<LPR>(r, sub, x);
        }
        s = lanes_sum<LPR>(s);
        if (ok) prolong(v, S.noff, fine, r.id, xi + r.om * (bi - (r.dg * xi - s)), sub, LPR, xf);
    });
}

// The same on the finest level: z, and this thread's parts of z.r and z.q.
template <int LPR>
__device__ void pass_top(const HierView &v, const Share &S, const double *r_, const double *q_, const double *x, double *z,
                         double &rz, double &zq) {
    for_items<LPR>(S.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        double xi = 0.0, bi = 0.0, qi = 0.0;
        if (ok) {
            r = share_row(v, S, k);
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
template <int LPR>
__device__ void pass_sweep(const HierView &v, const Share &S, const double *bl, const double *x, double *xo) {
    for_items<LPR>(S.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0;
        Row r{};
        if (ok) {
            r = share_row(v, S, k);
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
template <int LPR, bool FUSED>
__device__ void pass_product(const HierView &v, const Share &S, const double *z, const double *pold, double beta,
                             double *p, double *q, double &pq) {
    for_items<LPR>(S.nrow, [&](bool ok, int sub, int k) {
        double s = 0.0, pi = 0.0;
        Row r{};
        if (ok) {
            r = share_row(v, S, k);
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

// ---- block 0's levels

// Levels ng .. nlev - 1 on the right-hand side in v.b, the correction added to
// the x of level ng - 1.
__device__ void tier_cycle(const HierView &v, Shared &sh) {
    const int t0 = sh.ng, t1 = sh.nlev - 1;
    {
        Tier &T = sh.tier[t0];
        for (int i = threadIdx.x; i < T.n; i += kNT) {
            const double b = v.b[T.noff + i];
            T.b[i] = b;
            T.x[i] = T.om[i] * b;
        }
    }
    __syncthreads();
    for (int t = t0; t < t1; ++t) {
        const Tier &T = sh.tier[t], &C = sh.tier[t + 1];
        WITH_LANES(T.lprg, (for_items<LPR>(T.ng, [&](bool ok, int sub, int g) {
                       double s = 0.0;
                       if (ok)
                           for (int k = T.gs[g]; k < T.gs[g + 1]; ++k) {
                               const Row r = tier_row(v, T, T.own[k]);
                               if (sub == 0) s += T.b[r.id] - r.dg * T.x[r.id];
                               s += lane_dot<LPR>(r, sub, T.x);
                           }
                       s = lanes_sum<LPR>(s);
                       if (ok && sub == 0) {
                           C.b[g] = s;
                           C.x[g] = C.om[g] * s;
                       }
                   })));
        __syncthreads();
    }
    const Tier &Z = sh.tier[t1];
    const double *xz = Z.x;
    if (sh.dense) {
        for_items<8>(Z.n, [&](bool ok, int sub, int i) {
            double s = 0.0;
            if (ok)
                for (int j = sub; j < Z.n; j += 8) s += sh.inv[i * kDense + j] * Z.b[j];
            s = lanes_sum<8>(s);
            if (ok && sub == 0) Z.x[i] = s;
        });
        __syncthreads();
    } else {
        for (int k = 0; k < sh.sweeps; ++k) {
            const double *x = (k & 1) ? sh.alt : Z.x;
            double *xo = (k & 1) ? Z.x : sh.alt;
            WITH_LANES(Z.lpr, (for_items<LPR>(Z.n, [&](bool ok, int sub, int i) {
                           double s = 0.0;
                           Row r{};
                           if (ok) {
                               r = tier_row(v, Z, i);
                               s = lane_dot<LPR>(r, sub, x);
                           }
                           s = lanes_sum<LPR>(s);
                           if (ok && sub == 0) xo[i] = x[i] + r.om * (Z.b[i] - (r.dg * x[i] - s));
                       })));
            __syncthreads();
        }
    }
    // up: the coarsest level prolongs as it is, the others after their sweep
    for (int t = t1; t >= t0; --t) {
        const Tier &T = sh.tier[t];
        const bool top = t == t0;
        const int64_t fine = top ? sh.lev[t0 - 1].noff : 0;
        double *xf = top ? v.x + fine : sh.tier[t - 1].x;
        const int *of = top ? nullptr : sh.tier[t - 1].own, *gf = top ? nullptr : sh.tier[t - 1].gs;
        WITH_LANES(T.lpr, (for_items<LPR>(T.n, [&](bool ok, int sub, int i) {
                       double val = 0.0;
                       if (t == t1) {
                           if (ok) val = xz[i];
                       } else {
                           double s = 0.0;
                           Row r{};
                           if (ok) {
                               r = tier_row(v, T, i);
                               s = lane_dot<LPR>(r, sub, T.x);
                           }
                           s = lanes_sum<LPR>(s);
                           if (ok) val = T.x[i] + r.om * (T.b[i] - (r.dg * T.x[i] - s));
                       }
                       if (!ok) return;
                       if (top)
                           prolong(v, T.noff, fine, i, val, sub, LPR, xf);
                       else
                           for (int k = gf[i] + sub; k < gf[i + 1]; k += LPR) xf[of[k]] += val;
                   })));
        __syncthreads();
    }
}

// ---- shared-memory copies

// Block b's share of level l: its description, and its rows while they fit.
__device__ void load_share(const HierView &v, Shared &sh, int l, bool coarsest, unsigned b, unsigned nb, unsigned char *&p,
                           const unsigned char *end) {
    const LevelInfo &L = v.H->L[l];
    Share &S = sh.lev[l];
    const Seg g = coarsest ? Seg{} : v.seg[l * kMaxCtas + b];
    const int ch = (L.n + static_cast<int>(nb) - 1) / static_cast<int>(nb);
    const int c0 = min(L.n, static_cast<int>(b) * ch), c1 = min(L.n, c0 + ch);
    __syncthreads();
    if (threadIdx.x == 0) {
        S.noff = L.noff;
        S.n = L.n;
        S.whole = coarsest ? 1 : 0;
        S.first = coarsest ? c0 : g.m0;
        S.lfirst = g.l0;
        S.mlen = coarsest ? c1 - c0 : g.mlen;
        S.nrow = coarsest ? c1 - c0 : g.mlen + g.llen;
        S.g0 = g.g0;
        S.ngrp = g.glen;
        S.cached = 0;
        const double mean = static_cast<double>(L.nnz) / (L.n > 0 ? L.n : 1);
        S.lpr = lanes_for_items((L.n + nb - 1) / nb, mean);
        const int nco = coarsest ? L.n : v.H->L[l + 1].n;
        S.lprg = lanes_for_items((nco + nb - 1) / nb, mean * L.n / (nco > 0 ? nco : 1));
    }
    __syncthreads();
    const int nrow = S.nrow;
    int mine = 0;
    for (int k = threadIdx.x; k < nrow; k += kNT) mine += share_row(v, S, k).len;
    int ents;
    scan_nt(mine, sh.tmp, ents);
    const int64_t noff2 = L.noff + L.n;
    const size_t need = static_cast<size_t>(ents) * 12 + static_cast<size_t>(nrow) * 24 +
                        static_cast<size_t>(S.ngrp) * 4 + 8 * 16 + 16;
    if (static_cast<size_t>(end - p) < need) return;  // block-uniform
    double *w = reinterpret_cast<double *>(take(p, sizeof(double) * ents));
    double *dg = reinterpret_cast<double *>(take(p, sizeof(double) * nrow));
    double *om = reinterpret_cast<double *>(take(p, sizeof(double) * nrow));
    int *col = reinterpret_cast<int *>(take(p, sizeof(int) * ents));
    int *id = reinterpret_cast<int *>(take(p, sizeof(int) * nrow));
    int *off = reinterpret_cast<int *>(take(p, sizeof(int) * (nrow + 1)));
    int *gst = reinterpret_cast<int *>(take(p, sizeof(int) * (S.ngrp + 1)));
    int run = 0;
    for (int base = 0; base < nrow; base += kNT) {
        const int k = base + threadIdx.x;
        Row r{};
        if (k < nrow) r = share_row(v, S, k);
        int tot;
        const int at = scan_nt(r.len, sh.tmp, tot);
        if (k < nrow) {
            id[k] = r.id;
            dg[k] = r.dg;
            om[k] = r.om;
            off[k] = run + at;
        }
        run += tot;
    }
    if (threadIdx.x == 0) off[nrow] = run;
    for (int i = threadIdx.x; i < S.ngrp; i += kNT) {
        const int g0 = v.gs[noff2 + S.g0 + i] - S.first;
        gst[i] = g0;
        if (i == S.ngrp - 1) gst[i + 1] = g0 + v.gc[noff2 + S.g0 + i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < nrow; k += kNT / 32) {
        const int64_t e = v.rs[S.noff + id[k]];
        for (int q = lane; q < off[k + 1] - off[k]; q += 32) {
            col[off[k] + q] = v.ecol[e + q];
            w[off[k] + q] = v.ew[e + q];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        S.id = id;
        S.off = off;
        S.col = col;
        S.gst = gst;
        S.w = w;
        S.dg = dg;
        S.om = om;
        S.cached = 1;
    }
    __syncthreads();
}

// Block 0's level t (t >= ng): node arrays always in shared memory, entries while they fit.
__device__ void load_tier(const HierView &v, Shared &sh, int t, unsigned char *&p, const unsigned char *end) {
    const LevelInfo &L = v.H->L[t];
    Tier &T = sh.tier[t];
    const bool last = t == sh.nlev - 1;
    const int n = L.n, ng = last ? 0 : v.H->L[t + 1].n, nmem = last ? 0 : L.nmem;
    const int64_t noff = L.noff, noff2 = noff + n;
    double *dg = reinterpret_cast<double *>(take(p, sizeof(double) * n));
    double *om = reinterpret_cast<double *>(take(p, sizeof(double) * n));
    double *x = reinterpret_cast<double *>(take(p, sizeof(double) * n));
    double *b = reinterpret_cast<double *>(take(p, sizeof(double) * n));
    int *off = reinterpret_cast<int *>(take(p, sizeof(int) * (n + 1)));
    int *own = reinterpret_cast<int *>(take(p, sizeof(int) * nmem));
    int *gs = reinterpret_cast<int *>(take(p, sizeof(int) * (ng + 1)));
    const int ents = static_cast<int>(L.nnz);
    const bool fit = static_cast<size_t>(end - p) >= static_cast<size_t>(ents) * 12 + 64;
    double *w = fit ? reinterpret_cast<double *>(take(p, sizeof(double) * ents)) : nullptr;
    int *col = fit ? reinterpret_cast<int *>(take(p, sizeof(int) * ents)) : nullptr;
    int run = 0;
    for (int base = 0; base < n; base += kNT) {
        const int i = base + threadIdx.x;
        const int len = i < n ? v.rl[noff + i] : 0;
        int tot;
        const int at = scan_nt(len, sh.tmp, tot);
        if (i < n) {
            off[i] = run + at;
            dg[i] = v.dg[noff + i];
            om[i] = v.om[noff + i];
        }
        run += tot;
    }
    if (threadIdx.x == 0) off[n] = run;
    for (int k = threadIdx.x; k < nmem; k += kNT) own[k] = v.own[noff + k];
    for (int g = threadIdx.x; g < ng; g += kNT) gs[g] = v.gs[noff2 + g];
    if (threadIdx.x == 0) gs[ng] = nmem;
    __syncthreads();
    if (fit) {
        const int lane = threadIdx.x & 31;
        for (int i = threadIdx.x >> 5; i < n; i += kNT / 32) {
            const int64_t e = v.rs[noff + i];
            for (int q = lane; q < off[i + 1] - off[i]; q += 32) {
                col[off[i] + q] = v.ecol[e + q];
                w[off[i] + q] = v.ew[e + q];
            }
        }
    }
    if (threadIdx.x == 0) {
        T.noff = noff;
        T.n = n;
        T.ng = ng;
        const double mean = static_cast<double>(L.nnz) / (n > 0 ? n : 1);
        T.lpr = lanes_for_items(n, mean);
        T.lprg = lanes_for_items(ng, ng > 0 ? mean * n / ng : 1.0);
        T.cached = fit ? 1 : 0;
        T.off = off;
        T.own = own;
        T.gs = gs;
        T.col = col;
        T.w = w;
        T.dg = dg;
        T.om = om;
        T.x = x;
        T.b = b;
    }
    __syncthreads();
}

// ---- one V-cycle: x of the finest level holds om r on entry; alt is a free
// vector of the finest level's size.  Returns this thread's parts of z.r, z.q.
__device__ bool vcycle(const PcgArgs &a, Shared &sh, GridBar &bar, double *alt, double &rz, double &zq) {
    const HierView &v = a.v;
    const int nlev = sh.nlev, ng = sh.ng;
    const int nd = ng < nlev ? ng : nlev - 1;  // shared levels that are aggregated
    for (int l = 0; l < nd; ++l) {
        const Share &S = sh.lev[l];
        const int64_t noff2 = S.noff + S.n;
        WITH_LANES(S.lprg, (pass_down<LPR>(v, S, l ? v.b + S.noff : a.r, v.x + S.noff, noff2, v.b + noff2, v.x + noff2)));
        if (!bar.sync()) return false;
    }
    if (ng < nlev) {
        if (blockIdx.x == 0) tier_cycle(v, sh);
        if (!bar.sync()) return false;
    } else {
        const Share &S = sh.lev[nlev - 1];
        double *x = v.x + S.noff;
        const double *bl = nlev > 1 ? v.b + S.noff : a.r;
        if (sh.dense) {  // a finest level of at most kDense nodes (one block)
            for_items<8>(S.nrow, [&](bool ok, int sub, int k) {
                double s = 0.0;
                if (ok)
                    for (int j = sub; j < S.n; j += 8) s += v.H->inv[(S.first + k) * kDense + j] * bl[j];
                s = lanes_sum<8>(s);
                if (ok && sub == 0) x[S.first + k] = s;
            });
            if (!bar.sync()) return false;
        } else {
            for (int k = 0; k < sh.sweeps; ++k) {
                WITH_LANES(S.lpr, (pass_sweep<LPR>(v, S, bl, (k & 1) ? alt : x, (k & 1) ? x : alt)));
                if (!bar.sync()) return false;
            }
        }
        if (nlev == 1) {
            for (int k = threadIdx.x; k < S.nrow; k += kNT) {
                const int i = S.first + k;
                const double zi = x[i];
                a.z[i] = zi;
                rz += zi * a.r[i];
                zq += zi * a.q[i];
            }
            return true;
        }
        const int64_t fine = sh.lev[nlev - 2].noff;
        for (int k = threadIdx.x; k < S.nrow; k += kNT)
            prolong(v, S.noff, fine, S.first + k, x[S.first + k], 0, 1, v.x + fine);
        if (!bar.sync()) return false;
    }
    for (int l = nd - 1; l > 0; --l) {
        const Share &S = sh.lev[l];
        const int64_t fine = sh.lev[l - 1].noff;
        WITH_LANES(S.lpr, (pass_up<LPR>(v, S, v.b + S.noff, v.x + S.noff, fine, v.x + fine)));
        if (!bar.sync()) return false;
    }
    const Share &S = sh.lev[0];
    WITH_LANES(S.lpr, (pass_top<LPR>(v, S, a.r, a.q, v.x, a.z, rz, zq)));
    return true;
}

__global__ void __launch_bounds__(kSolveThreads, 1) k_pcg(PcgArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Shared sh;
    const HierView &v = a.v;
    Hier *H = v.H;
    const unsigned b = blockIdx.x, nb = gridDim.x;
    const int tid = threadIdx.x;
    GridBar bar(&H->bar[a.vcycle ? 3 : 1 + a.which], &H->err, nb);
    if (__syncthreads_or(H->err)) return;  // an earlier barrier failed: nothing here can be relied on

    // levels, and the rows of this block
    if (tid == 0) {
        sh.nlev = H->nlev;
        sh.dense = H->dense;
        sh.sweeps = H->sweeps;
        int ng = 0;
        while (ng < sh.nlev && H->L[ng].grid) ++ng;
        sh.ng = ng;
    }
    __syncthreads();
    unsigned char *p = smem;
    const unsigned char *end = smem + kSolveSmem;
    if (b == 0 && sh.ng < sh.nlev) {
        double *inv = reinterpret_cast<double *>(take(p, sizeof(double) * kDense * kDense));
        if (sh.dense)
            for (int i = tid; i < kDense * kDense; i += kNT) inv[i] = H->inv[i];
        double *alt = reinterpret_cast<double *>(take(p, sh.dense ? 0 : sizeof(double) * H->L[sh.nlev - 1].n));
        if (tid == 0) {
            sh.inv = inv;
            sh.alt = alt;
        }
        for (int t = sh.ng; t < sh.nlev; ++t) load_tier(v, sh, t, p, end);
    }
    for (int l = 0; l < sh.ng; ++l) load_share(v, sh, l, l == sh.nlev - 1, b, nb, p, end);
    const Share &S0 = sh.lev[0];

    const double trz = a.tol.rz_rel * a.scal[0];
    const double tres = fmax(a.tol.res_rel * a.scal[1], a.tol.res_floor);
    const int done_before = a.st->total;
    double *pbuf[2] = {a.p0, a.p1};
    // the residual of the start, in the sign-flipped unknowns (S: +1 rows, -1 columns)
    if (!a.vcycle) {
        for_items<8>(S0.nrow, [&](bool ok, int sub, int k) {
            double s = 0.0;
            Row r{};
            if (ok) {
                r = share_row(v, S0, k);
                if (a.schur) {
                    for (int64_t q = a.col_ptr[r.id] + sub; q < a.col_ptr[r.id + 1]; q += 8) {
                        const int32_t i = a.csc_row[q];
                        s += a.a2c[q] * (a.rhs[i] / a.diag[i]);
                    }
                    if (sub == 0) s -= a.rhs[a.nc + r.id];
                } else if (sub == 0) {
                    s = r.id < a.nc ? a.rhs[r.id] : -a.rhs[r.id];
                }
                if (a.which) {
                    s += lane_dot<8>(r, sub, a.d);
                    if (sub == 0) s -= r.dg * a.d[r.id];
                }
            }
            s = lanes_sum<8>(s);
            if (ok && sub == 0) {
                a.r[r.id] = s;
                v.x[r.id] = r.om * s;
                a.p0[r.id] = 0.0;
                a.q[r.id] = 0.0;
                if (!a.which) a.d[r.id] = 0.0;
            }
        });
    } else {
        for (int k = tid; k < S0.nrow; k += kNT) {
            const Row r = share_row(v, S0, k);
            v.x[r.id] = r.om * a.r[r.id];
        }
    }
    if (!bar.sync()) return;
    double rz_t = 0.0, zq_t = 0.0;
    if (!vcycle(a, sh, bar, a.p1, rz_t, zq_t)) return;
    if (a.vcycle) return;
    block_partials(sh, 1, rz_t, 0.0, 0.0);
    if (tid == 0) H->part[1][b] = sh.out[0];
    if (!bar.sync()) return;
    grid_totals(sh, H, 1, 1, nb);
    double rz = sh.out[0], beta = 0.0, res_max = INFINITY;
    int it = 0, conv = rz == 0.0 ? 1 : 0;
    const int left = a.tol.max_total - done_before;
    const int cap = max(1, min(a.tol.max_iter, left));
    const bool fused = a.e0 <= kFuseEntries * nb;
    while (!conv && it < cap) {
        ++it;
        const double *pold = pbuf[(it + 1) & 1];
        double *pn = pbuf[it & 1];
        double pq_t = 0.0;
        if (fused) {
            WITH_LANES(S0.lpr, (pass_product<LPR, true>(v, S0, a.z, pold, beta, pn, a.q, pq_t)));
        } else {
            for (int k = tid; k < S0.nrow; k += kNT) {
                const int i = S0.cached ? S0.id[k] : share_row(v, S0, k).id;
                pn[i] = a.z[i] + beta * pold[i];
            }
            if (!bar.sync()) return;
            WITH_LANES(S0.lpr, (pass_product<LPR, false>(v, S0, a.z, pold, beta, pn, a.q, pq_t)));
        }
        block_partials(sh, 1, pq_t, 0.0, 0.0);
        if (tid == 0) H->part[0][b] = sh.out[0];
        if (!bar.sync()) return;
        grid_totals(sh, H, 0, 1, nb);
        const double pq = sh.out[0];
        const double alpha = pq > 0.0 ? rz / pq : 0.0;
        double mx_t = 0.0;
        for (int k = tid; k < S0.nrow; k += kNT) {
            const Row r = share_row(v, S0, k);
            const int i = r.id;
            a.d[i] += alpha * pn[i];
            const double ri = a.r[i] - alpha * a.q[i];
            a.r[i] = ri;
            v.x[i] = r.om * ri;
            const double bt = a.schur ? a.volphi[i] : (i < a.nc ? a.b_row[i] : a.volphi[i - a.nc]);
            mx_t = fmax(mx_t, fabs(ri) / bt);
        }
        if (!bar.sync()) return;
        rz_t = zq_t = 0.0;
        if (!vcycle(a, sh, bar, const_cast<double *>(pold), rz_t, zq_t)) return;
        block_partials(sh, 3, rz_t, zq_t, mx_t);
        if (tid < 3) H->part[1 + tid][b] = sh.out[tid];
        if (!bar.sync()) return;
        grid_totals(sh, H, 1, 3, nb);
        // z.(r - r_old) = -alpha z.q: the flexible (Polak-Ribiere) beta
        beta = rz > 0.0 ? fmax(0.0, -alpha * sh.out[1] / rz) : 0.0;
        rz = sh.out[0];
        res_max = sh.out[2];
        conv = ((rz <= trz && res_max <= tres) || !(pq > 0.0) || !(rz > 0.0)) ? 1 : 0;
    }
    // back to the unknowns of rows and columns
    if (a.schur) {
        const int64_t ch = (a.nc + nb - 1) / nb;
        const int64_t i0 = b * ch, i1 = i0 + ch < a.nc ? i0 + ch : a.nc;
        for (int64_t i = i0 + tid; i < i1; i += kNT) {
            double s = a.rhs[i];
            for (int64_t e = a.row_ptr[i]; e < a.row_ptr[i + 1]; ++e) s += a.a2[e] * a.d[a.col[e]];
            a.dy[i] = s / a.diag[i];
            a.dy[a.nc + i] = -a.d[i];
        }
    } else {
        const int64_t n = 2 * a.nc, ch = (n + nb - 1) / nb;
        const int64_t i0 = b * ch, i1 = i0 + ch < n ? i0 + ch : n;
        for (int64_t i = i0 + tid; i < i1; i += kNT) a.dy[i] = i < a.nc ? a.d[i] : -a.d[i];
    }
    if (b == 0 && tid == 0) {
        a.st->rz = rz;
        a.st->res_max = res_max;
        a.st->iters = it;
        a.st->converged = conv;
        a.st->total = done_before + it;
    }
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
    double **dst[] = {&a.d, &a.r, &a.p0, &a.p1, &a.q, &a.z};
    for (double **d : dst) {
        *d = w;
        w += A.n0;
    }
    a.b_row = ptr<double>(m->bloc);
    a.volphi = ptr<double>(m->volphi);
    a.st = ptr<SolveStat>(A.stat);
    return a;
}

static void launch_pcg(bchar_mesh_t m, const PcgArgs &a) {
    static bool attrs = false;  // the shared-memory opt-in (harmless to repeat)
    if (!attrs) {
        cudaFuncSetAttribute(k_pcg, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSolveSmem));
        attrs = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(solve_grid(m->amg.e0));
    cfg.blockDim = dim3(kSolveThreads);
    cfg.dynamicSmemBytes = kSolveSmem;
    cfg.stream = m->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_pcg, a);
    ++m->launches;
}

void pcg_launch(bchar_mesh_t m, int which, const double *scal, const SolveTol &tol) {
    PcgArgs a = pcg_args(m);
    a.scal = scal;
    a.tol = tol;
    a.which = which;
    launch_pcg(m, a);
}

void amg_vcycle_once(bchar_mesh_t m) {
    PcgArgs a = pcg_args(m);
    a.scal = ptr<double>(m->partials);  // unused by a V-cycle
    a.vcycle = 1;
    cudaMemsetAsync(&ptr<Hier>(m->amg.hier)->bar[3], 0, sizeof(unsigned), m->stream);
    launch_pcg(m, a);
}

void amg_smooth_once(bchar_mesh_t m) {
    const PcgArgs a = pcg_args(m);
    k_level_sweep<<<blocks_for(a.n0), kThreads, 0, m->stream>>>(a.v, a.n0, a.r, a.z, a.q);
    ++m->launches;
}

}  // namespace bchar
