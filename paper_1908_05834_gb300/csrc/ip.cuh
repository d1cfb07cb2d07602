// The interior point's passes over the matrix entries and the constraint nodes
// (see launch_minimise for the problem and its symbols), each by all blocks of a
// cooperative launch: block b takes a range of rows, with their entries, and the
// same range of columns.
//
// The passes are bound by FP64 divisions and latency on small meshes and by
// memory on large ones; a row's entries are shared by LPR lanes.  Reciprocals of
// f, u and the multipliers are formed once per entry and pass (a division is
// about twelve instructions of a pipe that takes 19 clocks for each), and maxima
// are compared as integers (non-negative doubles order like their bits, and any
// negative one is below them).
#pragma once

#include "amg.cuh"
#include "gridbar.cuh"

namespace bchar {

// Scalars of the interior point, on the device.
struct IpScalars {
    double mu;          // mean complementarity (the solves read it and rp_max)
    double rp_max;      // max_l |rp_l| / b_l (the scaled constraint residual)
    double rd_max;      // max_e |rd_e|
    double rpq_max;     // max_l of the stationarity residuals of p and n
    double dual_max;    // max(max_l |y_l| b_l, max zl, max zh)
    double comp;        // sum of the complementarity products of all pairs
    double ap, ad;      // largest primal / dual step to the boundary (<= 1)
    int it;             // iterations done
    int cg;             // conjugate-gradient iterations of all solves so far (with the multigrid)
    int converged;
    int stop;           // no further iteration: converged, or at a cap
    int err;            // a grid barrier's wait ran out
    int levels, coarsest;  // the last hierarchy: levels, nodes of the coarsest
    unsigned bar;       // barrier counter of k_ip
};

static_assert(sizeof(IpScalars) <= kIpScalarBytes, "room in the host's copies");

// After the conjugate gradients' scalars in their buffer.
inline IpScalars *ip_scalars(bchar_mesh_t m) { return reinterpret_cast<IpScalars *>(ptr<CgState>(m->cg) + 1); }

// Blocks of a kernel of these passes alone (k_ip): one per 64 rows, and never more
// than the device holds at once, because a cooperative launch beyond that is refused.
inline int ip_grid(int64_t nc, int resident) {
    const int64_t most = resident < kMaxCtas ? resident : kMaxCtas, want = (nc + 63) / 64;
    return static_cast<int>(want < 1 || most < 1 ? 1 : (want < most ? want : most));
}

struct IpArgs {
    int64_t nc, nnz;
    const int64_t *row_ptr, *col_ptr;
    const int32_t *col, *csc_src;
    const double *a, *b_row, *volphi;
    double eps2, gamma, pairs, mu_floor, step;
    double qp_tol, mu_tol, rd_rel;  // stopping rule
    int max_it, max_cg;
    double *y, *f, *u, *zl, *zh, *p, *n, *zp, *zn;  // the iterate
    double *rp, *D, *q, *cl, *ch, *df, *du, *dzl, *dzh, *cp, *cn, *dp, *dn, *dzp, *dzn, *rhs, *dy;
    double *a2, *a2c, *diag, *exc, *g, *t;          // normal equations (g, t: with the rows eliminated, else null)
    double *part;                                   // 5 x kMaxCtas partial sums and maxima
    IpScalars *st;
};

__device__ __forceinline__ long long sbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ long long max_s(long long a, long long b) { return a > b ? a : b; }

// Items r0 .. r1 - 1 of the block's range, LPR lanes each; f(ok, sub, item) may
// shuffle within a warp.
template <int LPR, class F> __device__ __forceinline__ void ip_items(int64_t r0, int64_t r1, F f) {
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = r0 + static_cast<int>(threadIdx.x >> 5) * (32 / LPR); i0 < r1; i0 += blockDim.x / LPR) {
        const int64_t i = i0 + lane / LPR;
        f(i < r1, lane % LPR, i);
    }
}

template <int LPR> __device__ __forceinline__ double ip_lanes(double s) {
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// The block's range of rows (and of columns).
__device__ __forceinline__ void ip_range(int64_t nc, unsigned b, unsigned nb, int64_t &r0, int64_t &r1) {
    const int64_t ch = (nc + nb - 1) / nb;
    r0 = b * ch < nc ? b * ch : nc;
    r1 = r0 + ch < nc ? r0 + ch : nc;
}

// The target b_l of constraint node l: |K_l|_phi-balanced row target for a
// row node, |M_j|_phi for a column node.
__device__ __forceinline__ double ip_target(const IpArgs &A, int64_t l) {
    return l < A.nc ? A.b_row[l] : A.volphi[l - A.nc];
}

// Normal-equation weights of the rows: D_e, a2_e = a_e^2 D_e,
// exc_l = b_l^2 (eps^2 + p_l / zp_l + n_l / zn_l), diag_l = sum a^2 D + exc_l; with
// the rows eliminated also g_e = a2_e / sqrt(diag_row), t_row = exc_row / diag_row.
template <int LPR> __device__ void ip_weights_rows(const IpArgs &A, int64_t r0, int64_t r1) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t i) {
        double s = 0.0;
        int64_t e0 = 0, e1 = 0;
        if (ok) {
            e0 = A.row_ptr[i];
            e1 = A.row_ptr[i + 1];
            for (int64_t e = e0 + sub; e < e1; e += LPR) {
                const double De = 1.0 / (1.0 + A.zl[e] / A.f[e] + A.zh[e] / A.u[e]);
                const double ae = A.a[e], w = ae * ae * De;
                A.D[e] = De;
                A.a2[e] = w;
                s += w;
            }
        }
        s = ip_lanes<LPR>(s);
        if (!ok) return;
        const double bl = A.b_row[i];
        const double x = bl * bl * (A.eps2 + A.p[i] / A.zp[i] + A.n[i] / A.zn[i]);
        const double d = s + x;
        if (sub == 0) {
            A.diag[i] = d;
            A.exc[i] = x;
        }
        if (A.g) {
            const double w = 1.0 / sqrt(d);
            for (int64_t e = e0 + sub; e < e1; e += LPR) A.g[e] = A.a2[e] * w;
            if (sub == 0) A.t[i] = x / d;
        }
    });
}

// The same of the columns, once the rows' are in place.
template <int LPR> __device__ void ip_weights_cols(const IpArgs &A, int64_t r0, int64_t r1) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t j) {
        double s = 0.0;
        if (ok)
            for (int64_t k = A.col_ptr[j] + sub; k < A.col_ptr[j + 1]; k += LPR) {
                const double w = A.a2[A.csc_src[k]];
                A.a2c[k] = w;
                s += w;
            }
        s = ip_lanes<LPR>(s);
        if (ok && sub == 0) {
            const int64_t l = A.nc + j;
            const double bl = A.volphi[j];
            const double x = bl * bl * (A.eps2 + A.p[l] / A.zp[l] + A.n[l] / A.zn[l]);
            A.diag[l] = s + x;
            A.exc[l] = x;
        }
    });
}

// Reduced right-hand side per entry for the predictor (corrector = 0) or the
// corrector (with the predictor's direction in df..dzh):
//   cl = target of f zl, ch = target of u zh, q = -rd + cl / f - ch / u + (zh / u) ru,
//   rd = f - 1 - a (y_i + y_j) - zl + zh, ru = 2 - f - u.
template <int LPR> __device__ __noinline__ void ip_q(const IpArgs &A, int64_t r0, int64_t r1, int corrector, double sigma_mu) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t i) {
        if (!ok) return;
        const double yi = A.y[i];
        for (int64_t e = A.row_ptr[i] + sub; e < A.row_ptr[i + 1]; e += LPR) {
            const double f = A.f[e], u = A.u[e], zl = A.zl[e], zh = A.zh[e];
            const double rd = f - 1.0 - A.a[e] * (yi + A.y[A.nc + A.col[e]]) - zl + zh;
            double lo = -f * zl, hi = -u * zh;
            if (corrector) {
                lo += sigma_mu - A.df[e] * A.dzl[e];
                hi += sigma_mu - A.du[e] * A.dzh[e];
            }
            A.cl[e] = lo;
            A.ch[e] = hi;
            A.q[e] = -rd + lo / f + (zh * (2.0 - f - u) - hi) / u;
        }
    });
}

// Per node: the targets of p zp and n zn, and
// rhs_l = rp_l - (A-hat (D q))_l - b_l (p/zp sp - n/zn sn),
// sp = -(gamma - b y - zp) + cp / p, sn = -(gamma + b y - zn) + cn / n.
__device__ __forceinline__ void ip_rhs_node(const IpArgs &A, int64_t l, double s, int corrector, double sigma_mu) {
    const double bl = ip_target(A, l), ys = A.y[l] * bl;
    const double p = A.p[l], n = A.n[l], zp = A.zp[l], zn = A.zn[l];
    double c_p = -p * zp, c_n = -n * zn;
    if (corrector) {
        c_p += sigma_mu - A.dp[l] * A.dzp[l];
        c_n += sigma_mu - A.dn[l] * A.dzn[l];
    }
    A.cp[l] = c_p;
    A.cn[l] = c_n;
    // p/zp sp = (p (zp - (gamma - ys)) + cp) / zp, and the same of n (gamma -+ ys first: it cancels)
    const double tp = (p * (zp - (A.gamma - ys)) + c_p) / zp, tn = (n * (zn - (A.gamma + ys)) + c_n) / zn;
    A.rhs[l] = A.rp[l] - s - bl * (tp - tn);
}

template <int LPR> __device__ __noinline__ void ip_rhs(const IpArgs &A, int64_t r0, int64_t r1, int corrector, double sigma_mu) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t i) {
        double s = 0.0, c = 0.0;
        if (ok) {
            for (int64_t e = A.row_ptr[i] + sub; e < A.row_ptr[i + 1]; e += LPR) s += A.a[e] * A.D[e] * A.q[e];
            for (int64_t k = A.col_ptr[i] + sub; k < A.col_ptr[i + 1]; k += LPR) {
                const int32_t e = A.csc_src[k];
                c += A.a[e] * A.D[e] * A.q[e];
            }
        }
        s = ip_lanes<LPR>(s);
        c = ip_lanes<LPR>(c);
        if (ok && sub < 2) ip_rhs_node(A, sub ? A.nc + i : i, sub ? c : s, corrector, sigma_mu);
    });
}

// Direction per entry and per node from dy (of the block's own rows and columns)
// and sgn dc_j = dy of column j (any block's), and the ratio tests: the largest
// steps <= 1 that keep f, u, p, n (primal) and the multipliers (dual) positive,
// as the bits of their reciprocals max(1, -dv / v).
template <int LPR>
__device__ void ip_dir(const IpArgs &A, int64_t r0, int64_t r1, const double *dc, double sgn, long long &ap_inv,
                       long long &ad_inv) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t i) {
        if (!ok) return;
        const double di = A.dy[i];
        for (int64_t e = A.row_ptr[i] + sub; e < A.row_ptr[i + 1]; e += LPR) {
            const double f = A.f[e], u = A.u[e], zl = A.zl[e], zh = A.zh[e];
            const double fi = 1.0 / f, ui = 1.0 / u;
            const double d_f = A.D[e] * (A.q[e] + A.a[e] * (di + sgn * dc[A.col[e]]));
            const double d_u = 2.0 - f - u - d_f;
            const double d_zl = (A.cl[e] - zl * d_f) * fi;
            const double d_zh = (A.ch[e] - zh * d_u) * ui;
            A.df[e] = d_f;
            A.du[e] = d_u;
            A.dzl[e] = d_zl;
            A.dzh[e] = d_zh;
            ap_inv = max_s(ap_inv, max_s(sbits(-d_f * fi), sbits(-d_u * ui)));
            ad_inv = max_s(ad_inv, max_s(sbits(-d_zl / zl), sbits(-d_zh / zh)));
        }
    });
    for (int half = 0; half < 2; ++half)
        for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
            const int64_t l = half ? A.nc + i : i;
            const double bl = ip_target(A, l), ys = A.y[l] * bl, dys = A.dy[l] * bl;
            const double p = A.p[l], n = A.n[l], zp = A.zp[l], zn = A.zn[l], cp = A.cp[l], cn = A.cn[l];
            const double pi = 1.0 / p, ni = 1.0 / n, zpi = 1.0 / zp, zni = 1.0 / zn;
            const double sp = -(A.gamma - ys - zp) + cp * pi, sn = -(A.gamma + ys - zn) + cn * ni;
            const double d_p = p * zpi * (sp + dys), d_n = n * zni * (sn - dys);
            const double d_zp = (cp - zp * d_p) * pi, d_zn = (cn - zn * d_n) * ni;
            A.dp[l] = d_p;
            A.dn[l] = d_n;
            A.dzp[l] = d_zp;
            A.dzn[l] = d_zn;
            ap_inv = max_s(ap_inv, max_s(sbits(-d_p * pi), sbits(-d_n * ni)));
            ad_inv = max_s(ad_inv, max_s(sbits(-d_zp * zpi), sbits(-d_zn * zni)));
        }
}

// Complementarity after the predictor's steps to the boundary.
__device__ __forceinline__ double ip_comp_aff(const IpArgs &A, int64_t r0, int64_t r1, double ap, double ad) {
    double s = 0.0;
    for (int64_t e = A.row_ptr[r0] + threadIdx.x; e < A.row_ptr[r1]; e += blockDim.x)
        s += (A.f[e] + ap * A.df[e]) * (A.zl[e] + ad * A.dzl[e]) + (A.u[e] + ap * A.du[e]) * (A.zh[e] + ad * A.dzh[e]);
    for (int half = 0; half < 2; ++half)
        for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
            const int64_t l = half ? A.nc + i : i;
            s += (A.p[l] + ap * A.dp[l]) * (A.zp[l] + ad * A.dzp[l]) + (A.n[l] + ap * A.dn[l]) * (A.zn[l] + ad * A.dzn[l]);
        }
    return s;
}

__device__ __forceinline__ void ip_update(const IpArgs &A, int64_t r0, int64_t r1, double ap, double ad) {
    for (int64_t e = A.row_ptr[r0] + threadIdx.x; e < A.row_ptr[r1]; e += blockDim.x) {
        A.f[e] += ap * A.df[e];
        A.u[e] += ap * A.du[e];
        A.zl[e] += ad * A.dzl[e];
        A.zh[e] += ad * A.dzh[e];
    }
    for (int half = 0; half < 2; ++half)
        for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
            const int64_t l = half ? A.nc + i : i;
            A.y[l] += ad * A.dy[l];
            A.p[l] += ap * A.dp[l];
            A.n[l] += ap * A.dn[l];
            A.zp[l] += ad * A.dzp[l];
            A.zn[l] += ad * A.dzn[l];
        }
}

struct IpResid {
    double comp = 0.0;
    long long rp = 0, rd = 0, rpq = 0, dual = 0;  // bits of non-negative maxima
};

// Node l with constraint sum s: the constraint residual
// rp_l = b_l - (A-hat f)_l - eps^2 b_l^2 y_l - b_l (p_l - n_l), the stationarity
// residuals gamma -+ b y - z of p and n, and their complementarity.
__device__ __forceinline__ void ip_resid_node(const IpArgs &A, int64_t l, double s, IpResid &R) {
    const double bl = ip_target(A, l), ys = A.y[l] * bl;
    const double p = A.p[l], n = A.n[l], zp = A.zp[l], zn = A.zn[l];
    const double r = bl - s - A.eps2 * bl * ys - bl * (p - n);
    A.rp[l] = r;
    R.rp = max_s(R.rp, sbits(fabs(r) / bl));
    R.rpq = max_s(R.rpq, max_s(sbits(fabs(A.gamma - ys - zp)), sbits(fabs(A.gamma + ys - zn))));
    R.dual = max_s(R.dual, sbits(fabs(ys)));
    R.comp += p * zp + n * zn;
}

// The starting point of the iterations: f = u = 1 with multipliers z, y = 0,
// p = n = v with multipliers g.
struct IpStart {
    double z, v, g;
};

// START: the starting point is written here and is not read back (a pass of its
// own over the arrays, and reading them, took a third of the time at 10^6 cells).
template <int LPR, bool START> __device__ void ip_residual(const IpArgs &A, int64_t r0, int64_t r1, const IpStart &S, IpResid &R) {
    ip_items<LPR>(r0, r1, [&](bool ok, int sub, int64_t i) {
        double s = 0.0, c = 0.0;
        if (ok && START) {
            for (int64_t e = A.row_ptr[i] + sub; e < A.row_ptr[i + 1]; e += LPR) {
                A.f[e] = 1.0;
                A.u[e] = 1.0;
                A.zl[e] = S.z;
                A.zh[e] = S.z;
                R.comp += S.z + S.z;
                s += A.a[e];
            }
            for (int64_t k = A.col_ptr[i] + sub; k < A.col_ptr[i + 1]; k += LPR) c += A.a[A.csc_src[k]];
            if (sub < 2) {
                const int64_t l = sub ? A.nc + i : i;
                A.y[l] = 0.0;
                A.p[l] = S.v;
                A.n[l] = S.v;
                A.zp[l] = S.g;
                A.zn[l] = S.g;
                R.dual = max_s(R.dual, sbits(S.z));
            }
        } else if (ok) {
            const double yi = A.y[i];
            for (int64_t e = A.row_ptr[i] + sub; e < A.row_ptr[i + 1]; e += LPR) {
                const double f = A.f[e], zl = A.zl[e], zh = A.zh[e], ae = A.a[e];
                const double rd = f - 1.0 - ae * (yi + A.y[A.nc + A.col[e]]) - zl + zh;
                R.rd = max_s(R.rd, sbits(fabs(rd)));
                R.dual = max_s(R.dual, max_s(sbits(zl), sbits(zh)));
                R.comp += f * zl + A.u[e] * zh;
                s += ae * f;
            }
            for (int64_t k = A.col_ptr[i] + sub; k < A.col_ptr[i + 1]; k += LPR) {
                const int32_t e = A.csc_src[k];
                c += A.a[e] * A.f[e];
            }
        }
        s = ip_lanes<LPR>(s);
        c = ip_lanes<LPR>(c);
        if (ok && sub < 2) ip_resid_node(A, sub ? A.nc + i : i, sub ? c : s, R);
    });
}

// ---- reductions over the grid

struct IpShared {
    double sum[32];
    long long mx[4][32];
    double out[5];
    double ap, ad, sigma_mu;
};

// The block's parts of a sum (slot 0) and of NM maxima (slots 1 .. NM, bits).
// Every block reads the slots of all blocks, so a slot may be written only behind
// a grid barrier that follows its last read:
//   ip_steps to ip_corrector: 1 and 2 were read with no barrier since; 0 is written;
//   ip_corrector to ip_steps: 0 was read; barriers follow (and 1 and 2 are written);
//   ip_steps to ip_step: 1 and 2 were read; the barrier behind the update precedes
//     the check, which writes all of them.
template <bool SUM, int NM>
__device__ void ip_partials(IpShared &S, double *part, double sum, const long long *mx) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    long long m[NM > 0 ? NM : 1];
#pragma unroll
    for (int k = 0; k < NM; ++k) m[k] = mx[k];
    for (int o = 16; o > 0; o >>= 1) {
        if (SUM) sum += __shfl_xor_sync(0xffffffffu, sum, o);
#pragma unroll
        for (int k = 0; k < NM; ++k) m[k] = max_s(m[k], __shfl_xor_sync(0xffffffffu, m[k], o));
    }
    __syncthreads();
    if (lane == 0) {
        S.sum[wid] = sum;
#pragma unroll
        for (int k = 0; k < NM; ++k) S.mx[k][wid] = m[k];
    }
    __syncthreads();
    if (wid <= NM) {  // a warp per slot
        if (wid == 0) {
            double s = SUM && lane < nw ? S.sum[lane] : 0.0;
            if (SUM)
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (SUM && lane == 0) part[blockIdx.x] = s;
        } else {
            long long v = lane < nw ? S.mx[wid - 1][lane] : 0;
            for (int o = 16; o > 0; o >>= 1) v = max_s(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == 0) part[wid * kMaxCtas + blockIdx.x] = __longlong_as_double(v);
        }
    }
}

// The totals of slots s0 .. s1 - 1 over the grid, after a grid barrier, in S.out.
__device__ __forceinline__ void ip_totals(IpShared &S, const double *part, int s0, int s1) {
    const int lane = threadIdx.x & 31, s = s0 + static_cast<int>(threadIdx.x >> 5);
    const unsigned nb = gridDim.x;
    if (s < s1) {
        double sum = 0.0;
        long long m = 0;
        for (unsigned q = lane; q < nb; q += 32) {
            const double v = *reinterpret_cast<const volatile double *>(part + s * kMaxCtas + q);
            if (s == 0) sum += v;
            else m = max_s(m, sbits(v));
        }
        for (int o = 16; o > 0; o >>= 1) {
            if (s == 0) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            else m = max_s(m, __shfl_xor_sync(0xffffffffu, m, o));
        }
        if (lane == 0) S.out[s] = s == 0 ? sum : __longlong_as_double(m);
    }
    __syncthreads();
}

// ---- the parts of an iteration (every block of the grid; false: a barrier failed)

constexpr int kIpLanes = 4;  // lanes per row: the rows of the recipes hold 3 to 7 entries in the mean

// Weights; the normal equations' right-hand side of the predictor or corrector.
template <class Bar>
static __device__ __noinline__ bool ip_weights(const IpArgs &A, Bar &bar, int64_t r0, int64_t r1) {
    ip_weights_rows<kIpLanes>(A, r0, r1);
    if (!bar.sync()) return false;
    ip_weights_cols<kIpLanes>(A, r0, r1);
    return true;
}

// The direction's steps to the boundary, S.ap and S.ad.
template <class Bar>
static __device__ __noinline__ bool ip_steps(const IpArgs &A, Bar &bar, IpShared &S, int64_t r0, int64_t r1,
                                         const double *dc, double sgn) {
    long long mx[2] = {sbits(1.0), sbits(1.0)};
    ip_dir<kIpLanes>(A, r0, r1, dc, sgn, mx[0], mx[1]);
    ip_partials<false, 2>(S, A.part, 0.0, mx);
    if (!bar.sync()) return false;
    ip_totals(S, A.part, 1, 3);
    if (threadIdx.x < 2) (threadIdx.x ? S.ad : S.ap) = 1.0 / S.out[1 + threadIdx.x];
    __syncthreads();
    return true;
}

// Mehrotra's centring target (comp_aff / comp)^3 mu, not below the floor, and
// the corrector's right-hand side.
template <class Bar>
static __device__ __noinline__ bool ip_corrector(const IpArgs &A, Bar &bar, IpShared &S, int64_t r0, int64_t r1) {
    ip_partials<true, 0>(S, A.part, ip_comp_aff(A, r0, r1, S.ap, S.ad), nullptr);
    if (!bar.sync()) return false;
    ip_totals(S, A.part, 0, 1);
    if (threadIdx.x == 0) {
        const double r = S.out[0] / A.st->comp;
        S.sigma_mu = fmax(fmin(1.0, r * r * r) * A.st->mu, A.mu_floor);
    }
    __syncthreads();
    ip_q<kIpLanes>(A, r0, r1, 1, S.sigma_mu);
    if (!bar.sync()) return false;
    ip_rhs<kIpLanes>(A, r0, r1, 1, S.sigma_mu);
    return true;
}

// Residuals of the iterate, the scalars and the stopping test; cg: the solves'
// conjugate-gradient iterations so far (of block 0), done: iterations done.
template <bool START, class Bar>
static __device__ __noinline__ bool ip_check(const IpArgs &A, Bar &bar, IpShared &S, int64_t r0, int64_t r1, int cg,
                                             int done, const IpStart &at) {
    IpResid R;
    ip_residual<kIpLanes, START>(A, r0, r1, at, R);
    const long long mx[4] = {R.rp, R.rd, R.rpq, R.dual};
    ip_partials<true, 4>(S, A.part, R.comp, mx);
    if (!bar.sync()) return false;
    if (blockIdx.x != 0) return true;
    ip_totals(S, A.part, 0, 5);
    if (threadIdx.x == 0) {
        IpScalars &st = *A.st;
        const double mu = S.out[0] / A.pairs;
        st.comp = S.out[0];
        st.mu = mu;
        st.rp_max = S.out[1];
        st.rd_max = S.out[2];
        st.rpq_max = S.out[3];
        st.dual_max = S.out[4];
        st.it = done;
        st.cg = cg;
        st.converged = S.out[1] <= A.qp_tol && mu <= A.mu_tol && S.out[2] <= A.rd_rel * (1.0 + S.out[4]) &&
                       S.out[3] <= A.rd_rel * (1.0 + A.gamma);
        st.stop = st.converged || done >= A.max_it || cg >= A.max_cg;
    }
    return true;
}

// The step, a fraction of the way to the boundary, then the check.
template <class Bar>
static __device__ __noinline__ bool ip_step(const IpArgs &A, Bar &bar, IpShared &S, int64_t r0, int64_t r1, int cg,
                                        int done) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.st->ap = S.ap;
        A.st->ad = S.ad;
    }
    ip_update(A, r0, r1, A.step * S.ap, A.step * S.ad);
    if (!bar.sync()) return false;
    return ip_check<false>(A, bar, S, r0, r1, cg, done, IpStart{});
}

}  // namespace bchar
