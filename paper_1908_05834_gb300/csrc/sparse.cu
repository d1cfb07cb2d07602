// FP64 matrix stages of a B-char step:
//   - device-wide scans (row / column pointers),
//   - the column view of A (deterministic: columns sorted by row),
//   - N alternating column/row scalings (Sec 3.2, eq. volAdj), kept as
//     diagonal factors, A^(N) = diag(R) A^(0) diag(C),
//   - the mass-conservation minimisation (Sec 3.2, eq. opti_masscons) with
//     its bounds 0 <= 1 + x <= 2 inside the problem and an elastic penalty on
//     the relative violations of the mass constraints (quadratic, weight
//     1/eps^2, up to 1e-6; linear beyond), by a primal-dual interior-point
//     method whose normal equations (A-hat D A-hat^T + diag(exc)) are the
//     bipartite matrix [[D_r, W], [W^T, D_c]], W_ij = a_ij^2 D_ij, applied
//     through the row and column views of A without forming A-hat and solved
//     by conjugate gradients with an aggregation-multigrid preconditioner,
//   - a final column scaling (global mass to rounding), W_KM = a_KM / |K|_phi
//     and the update c^{n+1} = W c^n (eq. phys-inter-ELLAM) with FP64
//     accumulation.
// All sums run in a fixed order (no floating-point atomics), so a step is
// bitwise reproducible.
#include <math.h>
#include <stddef.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <time.h>

#include "amg.cuh"
#include "device.cuh"
#include "ip.cuh"
#include "tiles.cuh"

namespace bchar {

#define GRID_STRIDE(i, n)                                                            \
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < (n); \
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)

// ---------------------------------------------------------------- scan

__global__ void k_scan_partial(const int32_t *in, int64_t n, int64_t *block_sums) {
    dep_enter();
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanChunk;
    int64_t s = 0;
    for (int i = threadIdx.x; i < kScanChunk; i += blockDim.x)
        if (base + i < n) s += in[base + i];
    __shared__ int64_t sh[kThreads];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) block_sums[blockIdx.x] = sh[0];
}

// One block: exclusive scan of nb block sums in place, total in sums[nb].
__global__ void k_scan_top(int64_t *sums, int nb) {
    dep_enter();
    __shared__ int64_t sh[1024];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += 1024) {
        int i = base + threadIdx.x;
        int64_t v = i < nb ? sums[i] : 0;
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {  // Hillis-Steele inclusive scan
            int64_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
            __syncthreads();
            sh[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) sums[i] = carry + sh[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == 0) carry += sh[1023];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void k_scan_final(const int32_t *in, int64_t n, const int64_t *block_off, int64_t *out, int nb) {
    dep_enter();
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanChunk;
    constexpr int per = kScanChunk / kThreads;
    const int64_t mine = base + static_cast<int64_t>(threadIdx.x) * per;
    int64_t local[per];
    int64_t s = 0;
    for (int k = 0; k < per; ++k) {
        local[k] = (mine + k < n) ? in[mine + k] : 0;
        s += local[k];
    }
    __shared__ int64_t sh[kThreads];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < kThreads; o <<= 1) {
        int64_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    int64_t run = block_off[blockIdx.x] + sh[threadIdx.x] - s;
    for (int k = 0; k < per; ++k) {
        if (mine + k < n) out[mine + k] = run;
        run += local[k];
    }
    if (blockIdx.x == nb - 1 && threadIdx.x == 0) out[n] = block_off[nb];
}

void scan_i32_to_i64(bchar_mesh_t m, const int32_t *in, int64_t *out, int64_t n) {
    const int nb = static_cast<int>((n + kScanChunk - 1) / kScanChunk);
    const int nbb = nb < 1 ? 1 : nb;
    ensure(m, m->scan_tmp, sizeof(int64_t) * (nbb + 1));
    int64_t *sums = ptr<int64_t>(m->scan_tmp);
    launch_dep(k_scan_partial, nbb, kThreads, m->stream, in, n, sums);
    launch_dep(k_scan_top, 1, 1024, m->stream, sums, nbb);
    launch_dep(k_scan_final, nbb, kThreads, m->stream, in, n, sums, out, nbb);
    m->launches += 3;
}

// ---------------------------------------------------------------- reductions

// Final reduction of per-block partial sums (fixed order) into *out.
__global__ void k_sum_partials(const double *partials, int n, double *out) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += partials[i];
    s = block_sum(s);
    if (threadIdx.x == 0) *out = s;
}

// ---------------------------------------------------------------- column view

__global__ void k_fill_columns(int64_t nc, const int64_t *row_ptr, const int32_t *col, const int64_t *col_ptr,
                               int32_t *fill, int32_t *csc_row, int32_t *csc_src) {
    GRID_STRIDE(i, nc) {
        for (int64_t e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int32_t j = col[e];
            const int64_t p = col_ptr[j] + atomicAdd(&fill[j], 1);
            csc_row[p] = static_cast<int32_t>(i);
            csc_src[p] = static_cast<int32_t>(e);
        }
    }
}

// Entries of each column in increasing row order (insertion sort; columns
// hold a few tens of entries at most).
__global__ void k_sort_columns(int64_t nc, const int64_t *col_ptr, int32_t *csc_row, int32_t *csc_src) {
    GRID_STRIDE(j, nc) {
        const int64_t b = col_ptr[j], e = col_ptr[j + 1];
        for (int64_t p = b + 1; p < e; ++p) {
            const int32_t r = csc_row[p], s = csc_src[p];
            int64_t q = p;
            while (q > b && csc_row[q - 1] > r) {
                csc_row[q] = csc_row[q - 1];
                csc_src[q] = csc_src[q - 1];
                --q;
            }
            csc_row[q] = r;
            csc_src[q] = s;
        }
    }
}

void launch_transpose(bchar_mesh_t m) {
    scan_i32_to_i64(m, ptr<int32_t>(m->colcnt), ptr<int64_t>(m->col_ptr), m->nc);
    cudaMemsetAsync(m->colfill.p, 0, sizeof(int32_t) * m->nc, m->stream);
    k_fill_columns<<<blocks_for(m->nc), kThreads, 0, m->stream>>>(m->nc, ptr<int64_t>(m->row_ptr), ptr<int32_t>(m->col),
                                                                  ptr<int64_t>(m->col_ptr), ptr<int32_t>(m->colfill),
                                                                  ptr<int32_t>(m->csc_row), ptr<int32_t>(m->csc_src));
    k_sort_columns<<<blocks_for(m->nc), kThreads, 0, m->stream>>>(m->nc, ptr<int64_t>(m->col_ptr),
                                                                  ptr<int32_t>(m->csc_row), ptr<int32_t>(m->csc_src));
    m->launches += 2;
}

// ---------------------------------------------------------------- sub-warp row walks
//
// The streaming stages (scalings, update) walk rows of a few to a few tens of
// entries: L lanes of a warp share one row (L a power of two sized to the mean
// row length), so consecutive lanes read consecutive entries and a warp reads
// 32 consecutive entries of neighbouring rows at once.  A row's partial sums
// are reduced by shuffles within its L lanes.  Every lane of a warp runs the
// same number of outer iterations (rows past the end contribute nothing), so
// the shuffles always see the whole warp.  The grid is persistent (a fixed
// multiple of the SM count), so the order of every sum is fixed.

template <int L> __device__ __forceinline__ double group_sum(double v) {
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Lanes per row for a mean of `mean` entries per row.
static int lanes_for(double mean) {
    int L = 2;
    while (L < 32 && L < mean) L <<= 1;
    return L;
}

#define DISPATCH_LANES(L, CALL)                 \
    switch (L) {                                \
    case 2: { constexpr int LL = 2; CALL; } break;   \
    case 4: { constexpr int LL = 4; CALL; } break;   \
    case 8: { constexpr int LL = 8; CALL; } break;   \
    case 16: { constexpr int LL = 16; CALL; } break; \
    default: { constexpr int LL = 32; CALL; } break; \
    }

constexpr int kStreamBlocks = 152 * 8;  // persistent grid of the streaming kernels (256 threads each)

// ---------------------------------------------------------------- tiles of the two views

template <class K> static void allow_tile_smem(K kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kTileSmem));
}

__global__ void k_tile_bounds(int64_t n, const int64_t *ptr, int64_t ntile, int32_t *tile) {
    GRID_STRIDE(k, ntile + 1) {
        if (k == ntile) {
            tile[k] = static_cast<int32_t>(n);
        } else {
            const int64_t want = k * static_cast<int64_t>(kTileEntries);
            int64_t lo = 0, hi = n;  // the first l in [0, n] with ptr[l] >= want
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (ptr[mid] >= want) hi = mid;
                else lo = mid + 1;
            }
            tile[k] = static_cast<int32_t>(lo);
        }
    }
}

__global__ void k_scale_tiles(LineView V, const double *f, const double *tgt, double *out);
__global__ void k_scaled_col_error(LineView V, const double *R, const double *C, const double *volphi,
                                   unsigned long long *slot);
__global__ void k_cg_matvec(LineView Vr, LineView Vc, const double *diag, const double *p, double *q,
                            double *partials, const CgState *st);
template <class T> __global__ void k_spmv(LineView V, const double *volphi, const T *c_in, T *c_out, double *partials);

void tiles_opt_in() {
    allow_tile_smem(k_scale_tiles);
    allow_tile_smem(k_scaled_col_error);
    allow_tile_smem(k_cg_matvec);
    allow_tile_smem(k_spmv<float>);
    allow_tile_smem(k_spmv<double>);
}

bool launch_tiles(bchar_mesh_t m) {
    m->ntile = tile_count(m->nnz);
    const size_t b = sizeof(int32_t) * (m->ntile + 1);
    if (!ensure(m, m->tile_r, b) || !ensure(m, m->tile_c, b)) return false;
    k_tile_bounds<<<blocks_for(m->ntile + 1), kThreads, 0, m->stream>>>(m->nc, ptr<int64_t>(m->row_ptr), m->ntile,
                                                                        ptr<int32_t>(m->tile_r));
    k_tile_bounds<<<blocks_for(m->ntile + 1), kThreads, 0, m->stream>>>(m->nc, ptr<int64_t>(m->col_ptr), m->ntile,
                                                                        ptr<int32_t>(m->tile_c));
    m->launches += 2;
    return true;
}

static LineView row_view(bchar_mesh_t m, const double *val) {
    return LineView{m->nc, ptr<int64_t>(m->row_ptr), ptr<int32_t>(m->col), val, ptr<int32_t>(m->tile_r), m->ntile};
}

static LineView col_view(bchar_mesh_t m, const double *val) {
    return LineView{m->nc, ptr<int64_t>(m->col_ptr), ptr<int32_t>(m->csc_row), val, ptr<int32_t>(m->tile_c), m->ntile};
}

static int tile_grid(int64_t ntiles) { return static_cast<int>(ntiles < kTileBlocks ? (ntiles > 0 ? ntiles : 1) : kTileBlocks); }

// ---------------------------------------------------------------- scaling (eq. volAdj)

__global__ void k_fill(double *v, int64_t n, double val) {
    GRID_STRIDE(i, n) v[i] = val;
}

// a0 in column order (a0c[p] = a0[csc_src[p]]), once per step, so that the
// column passes stream their values.
__global__ void k_gather_col_values(int64_t nnz, const int32_t *csc_src, const double *a0, double *a0c) {
    GRID_STRIDE(p, nnz) a0c[p] = a0[csc_src[p]];
}

// Line sums of one view: out_l = tgt_l / sum_k v_k f[idx_k] over line l (a
// column of the column view with f = R, or a row of the row view with f = C):
// a^{n+1/2}: C_j = |M_j|_phi / sum_i R_i a0_ij; a^{n+1}: R_i = b_i / sum_j a0_ij C_j.
struct ScaleEpi {
    const double *tgt;
    double *out;
    __device__ void operator()(int64_t l, double s) { out[l] = tgt[l] / s; }
};

struct NoEpi {
    __device__ void operator()(int64_t, double) {}
};

__global__ void __launch_bounds__(kTileThreads) k_scale_tiles(LineView V, const double *f, const double *tgt,
                                                              double *out) {
    extern __shared__ __align__(16) unsigned char smem[];
    ScaleEpi epi{tgt, out};
    NoEpi none;
    const LineView nov{0, nullptr, nullptr, nullptr, nullptr, 0};
    tile_loop(V, f, epi, nov, f, none, smem);
}

// aN = R a0 C per entry (row view)
template <int L>
__global__ void __launch_bounds__(256) k_apply_scaling(int64_t nc, const int64_t *row_ptr, const int32_t *col,
                                                       const double *a0, const double *R, const double *C,
                                                       double *aN) {
    constexpr int G = 256 / L;
    const int g = threadIdx.x / L, lane = threadIdx.x % L;
    for (int64_t base = static_cast<int64_t>(blockIdx.x) * G; base < nc; base += static_cast<int64_t>(gridDim.x) * G) {
        const int64_t i = base + g;
        if (i < nc) {
            const double ri = R[i];
            for (int64_t e = row_ptr[i] + lane; e < row_ptr[i + 1]; e += L) aN[e] = ri * a0[e] * C[col[e]];
        }
    }
}

// max_j |C_j sum_i R_i a0_ij - |M_j|_phi| / |M_j|_phi (the column sums of A^(N))
struct ColErrEpi {
    const double *C, *volphi;
    double mx;
    __device__ void operator()(int64_t j, double s) { mx = fmax(mx, fabs(C[j] * s - volphi[j]) / volphi[j]); }
};

__global__ void __launch_bounds__(kTileThreads) k_scaled_col_error(LineView V, const double *R, const double *C,
                                                                   const double *volphi, unsigned long long *slot) {
    extern __shared__ __align__(16) unsigned char smem[];
    ColErrEpi epi{C, volphi, 0.0};
    NoEpi none;
    const LineView nov{0, nullptr, nullptr, nullptr, nullptr, 0};
    tile_loop(V, R, epi, nov, R, none, smem);
    const double mx = block_max(epi.mx);
    if (threadIdx.x == 0) atomic_max_nonneg(slot, mx);
}

// max_j |sum_i a_ij - |M_j|_phi| / |M_j|_phi over the column view of a
__global__ void k_col_error(int64_t nc, const int64_t *col_ptr, const int32_t *csc_src, const double *a,
                            const double *volphi, unsigned long long *slot) {
    double mx = 0.0;
    GRID_STRIDE(j, nc) {
        double s = 0.0;
        for (int64_t p = col_ptr[j]; p < col_ptr[j + 1]; ++p) s += a[csc_src[p]];
        mx = fmax(mx, fabs(s - volphi[j]) / volphi[j]);
    }
    mx = block_max(mx);
    if (threadIdx.x == 0) atomic_max_nonneg(slot, mx);
}

static void scaling_pass(bchar_mesh_t m, bool col_pass, const double *a0c) {
    const int grid = tile_grid(m->ntile);
    if (col_pass)
        k_scale_tiles<<<grid, kTileThreads, kTileSmem, m->stream>>>(col_view(m, a0c), ptr<double>(m->R), ptr<double>(m->volphi),
                                                            ptr<double>(m->C));
    else
        k_scale_tiles<<<grid, kTileThreads, kTileSmem, m->stream>>>(row_view(m, ptr<double>(m->a0)), ptr<double>(m->C),
                                                            ptr<double>(m->bloc), ptr<double>(m->R));
    ++m->launches;
}

void launch_scaling(bchar_mesh_t m) {
    const int64_t nc = m->nc, nnz = m->nnz;
    const int L = lanes_for(static_cast<double>(nnz) / static_cast<double>(nc > 0 ? nc : 1));
    double *a0c = ptr<double>(m->a2c);  // scratch until the minimisation: A^(0) in column order
    k_gather_col_values<<<blocks_for(nnz), kThreads, 0, m->stream>>>(nnz, ptr<int32_t>(m->csc_src), ptr<double>(m->a0),
                                                                   a0c);
    k_fill<<<blocks_for(nc), kThreads, 0, m->stream>>>(ptr<double>(m->R), nc, 1.0);
    m->launches += 2;
    for (int it = 0; it < m->opt.n_scale; ++it) {
        scaling_pass(m, true, a0c);
        scaling_pass(m, false, a0c);
    }
    if (m->opt.n_scale == 0) {
        k_fill<<<blocks_for(nc), kThreads, 0, m->stream>>>(ptr<double>(m->C), nc, 1.0);
        ++m->launches;
    }
    DISPATCH_LANES(L, (k_apply_scaling<LL><<<kStreamBlocks, 256, 0, m->stream>>>(
                           nc, ptr<int64_t>(m->row_ptr), ptr<int32_t>(m->col), ptr<double>(m->a0), ptr<double>(m->R),
                           ptr<double>(m->C), ptr<double>(m->aN))));
    DevInfo *di = ptr<DevInfo>(m->dinfo);
    k_scaled_col_error<<<tile_grid(m->ntile), kTileThreads, kTileSmem, m->stream>>>(
        col_view(m, a0c), ptr<double>(m->R), ptr<double>(m->C), ptr<double>(m->volphi),
        reinterpret_cast<unsigned long long *>(&di->scale_err));
    m->launches += 2;
}

// One column and one row scaling (timing aid: the streaming stages of a step).
void launch_scaling_once(bchar_mesh_t m) {
    scaling_pass(m, true, ptr<double>(m->a2c));
    scaling_pass(m, false, ptr<double>(m->a2c));
}

// ---------------------------------------------------------------- minimisation
//
// eq. opti_masscons with the bounds 0 <= f = 1 + x <= 2 inside the problem and
// the 2 n_c mass constraints enforced by an elastic penalty on their relative
// violations v_l (see bchar_step in bchar.h): quadratic, weight 1/eps^2, up to
// |v| = 1e-6 and linear beyond, slope gamma = 1e-6 / eps^2.  Solved by a
// primal-dual interior-point method (Mehrotra predictor-corrector) with f, its
// upper slack u = 2 - f (carried separately: f near 2 would lose u to
// rounding), the bound multipliers zl, zh >= 0, the constraint multipliers y
// (node l < n_c: row l, node n_c + j: column j) and, per node, the violation
// beyond the quadratic zone split p - n with p, n >= 0 and multipliers zp, zn:
//     stationarity  rd_e = f_e - 1 - a_e (y_i + y_{n_c+j}) - zl_e + zh_e,
//                   gamma - b_l y_l - zp_l = 0,  gamma + b_l y_l - zn_l = 0
//     constraints   rp_l = b_l - (A-hat f)_l - eps^2 b_l^2 y_l - b_l (p_l - n_l)
//     slack         ru_e = 2 - f_e - u_e
// Each iteration solves the normal equations (A-hat D A-hat^T + diag(exc)) dy = r,
// D_e = 1 / (1 + zl_e / f_e + zh_e / u_e), exc_l = b_l^2 (eps^2 + p_l / zp_l +
// n_l / zn_l), twice with one preconditioner: the bipartite Laplacian of the
// step's pattern with edge weights a_e^2 D_e and that diagonal shift, by the
// conjugate gradients below with the aggregation multigrid.

// Preconditioned conjugate gradients on (A-hat A-hat^T + W) d = F.  Every
// kernel returns at once when the solve has converged, so that batches of
// iterations can be queued without reading the state back each time.

__global__ void k_copy(int64_t n, const double *in, double *out, const CgState *st) {
    if (st && st->converged) return;
    GRID_STRIDE(i, n) out[i] = in[i];
}

// res = rhs - q (the residual of a starting guess whose product is q)
__global__ void k_residual(int64_t n, const double *rhs, const double *q, double *res) {
    GRID_STRIDE(i, n) res[i] = rhs[i] - q[i];
}

// Clears the converged flag a finished solve left, before a product that the
// next solve's start needs (the CG kernels return at once while it is set).
__global__ void k_cg_reopen(CgState *st) { st->converged = 0; }

// z = res / diag (Jacobi preconditioner)
__global__ void k_jacobi_precond(int64_t n, const double *diag, const double *res, double *z, const CgState *st) {
    dep_enter();
    if (st && st->converged) return;
    GRID_STRIDE(i, n) z[i] = res[i] / diag[i];
}

__global__ void k_dot(int64_t n, const double *a, const double *b, double *partials, const CgState *st) {
    if (st && st->converged) return;
    double acc = 0.0;
    GRID_STRIDE(i, n) acc += a[i] * b[i];
    acc = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// Start of a solve: z.res of the initial residual, the two stopping targets
// (z.res <= target and max_l |res_l| / b_l <= target_res; the initial value of
// the latter is rhs_max).
__global__ void k_cg_start(const double *partials, int nparts, double target, double target_res, double rhs_max,
                           CgState *st) {
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += partials[i];
    s = block_sum(s);
    if (threadIdx.x == 0) {
        st->rz = s;
        st->target = target;
        st->target_res = target_res;
        st->res_max = rhs_max;
        st->converged = (s == 0.0) || (s <= target && rhs_max <= target_res);
        st->iters = 0;
    }
}

// q = (A-hat D A-hat^T + diag(exc)) p through the row view (node l < n_c:
// row l, its entries a2 = a^2 D against the column nodes) and the column view
// (node n_c + j: column j, its entries a2c against the row nodes), tile by
// tile (the row view's tiles first), and per-block partial sums of p.q.
struct MatvecEpi {
    const double *diag, *p;
    double *q;
    int64_t off;  // 0 for the rows, n_c for the columns
    double acc;
    __device__ void operator()(int64_t l, double s) {
        const int64_t node = off + l;
        const double v = s + diag[node] * p[node];
        q[node] = v;
        acc += p[node] * v;
    }
};

__global__ void __launch_bounds__(kTileThreads) k_cg_matvec(LineView Vr, LineView Vc, const double *diag,
                                                            const double *p, double *q, double *partials,
                                                            const CgState *st) {
    dep_enter();
    if (st->converged) return;
    extern __shared__ __align__(16) unsigned char smem[];
    const int64_t nc = Vr.n;
    MatvecEpi er{diag, p, q, 0, 0.0}, ec{diag, p, q, nc, 0.0};
    tile_loop(Vr, p + nc, er, Vc, p, ec, smem);
    const double acc = block_sum(er.acc + ec.acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

__global__ void k_cg_alpha(const double *partials, int nparts, CgState *st) {
    dep_enter();
    if (st->converged) return;
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += partials[i];
    s = block_sum(s);
    if (threadIdx.x == 0) {
        st->pq = s;
        st->alpha = s > 0.0 ? st->rz / s : 0.0;
    }
}

// d += alpha p, res -= alpha q (the previous residual kept in rp), per-block
// maxima of |res_l| / b_l (res is the constraint residual the direction leaves)
__global__ void k_cg_update(int64_t n2, const double *p, const double *q, double *d, double *res, double *rp,
                            const double *b_row, const double *volphi, double *partials, const CgState *st) {
    dep_enter();
    if (st->converged) return;
    const double alpha = st->alpha;
    const int64_t nc = n2 / 2;
    double mx = 0.0;
    GRID_STRIDE(l, n2) {
        d[l] += alpha * p[l];
        const double r0 = res[l];
        rp[l] = r0;
        const double r = r0 - alpha * q[l];
        res[l] = r;
        mx = fmax(mx, fabs(r) / (l < nc ? b_row[l] : volphi[l - nc]));
    }
    mx = block_max(mx);
    if (threadIdx.x == 0) partials[blockIdx.x] = mx;
}

// partial sums of z.res and z.rp (flexible, Polak-Ribiere form of beta: the
// preconditioner may differ slightly between applications)
__global__ void k_dot2(int64_t n, const double *z, const double *res, const double *rp, double *pa, double *pb,
                       const CgState *st) {
    dep_enter();
    if (st && st->converged) return;
    double a = 0.0, b = 0.0;
    GRID_STRIDE(i, n) {
        a += z[i] * res[i];
        b += z[i] * rp[i];
    }
    a = block_sum(a);
    b = block_sum(b);
    if (threadIdx.x == 0) {
        pa[blockIdx.x] = a;
        pb[blockIdx.x] = b;
    }
}

__global__ void k_cg_beta(const double *rz_parts, const double *zp_parts, const double *res_parts, int nparts,
                          CgState *st) {
    dep_enter();
    if (st->converged) return;
    double rz = 0.0, zp = 0.0, mx = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) {
        rz += rz_parts[i];
        zp += zp_parts[i];
        mx = fmax(mx, res_parts[i]);
    }
    rz = block_sum(rz);
    zp = block_sum(zp);
    mx = block_max(mx);
    if (threadIdx.x == 0) {
        st->beta = st->rz > 0.0 ? fmax(0.0, (rz - zp) / st->rz) : 0.0;
        st->rz = rz;
        st->res_max = mx;
        st->iters += 1;
        if ((rz <= st->target && mx <= st->target_res) || !(st->pq > 0.0) || !(rz > 0.0)) st->converged = 1;
    }
}

__global__ void k_cg_pupdate(int64_t n2, const double *z, double *p, const CgState *st) {
    dep_enter();
    if (st->converged) return;
    const double beta = st->beta;
    GRID_STRIDE(l, n2) p[l] = z[l] + beta * p[l];
}

// Parts of an iteration as one cooperative kernel each: the start of the
// minimisation, and the passes around solves that run as kernels of their own
// (qp_precond = 0; with the multigrid an iteration is the two kernels of amg.cu
// and pcg.cu).
enum IpPart { kIpStart, kIpBegin, kIpMid, kIpEnd };
constexpr int kIpThreads = 1024;  // one block per SM: at 10^6 cells the loads in flight bound it

__global__ void __launch_bounds__(kIpThreads, 1) k_ip(const __grid_constant__ IpArgs A, int part, IpStart at) {
    __shared__ IpShared S;
    const unsigned b = blockIdx.x, nb = gridDim.x;
    GridBar bar(&A.st->bar, &A.st->err, nb);
    int64_t r0, r1;
    ip_range(A.nc, b, nb, r0, r1);
    const int done = A.st->it;
    if (part == kIpStart) {
        ip_check<true>(A, bar, S, r0, r1, 0, 0, at);
    } else if (part == kIpBegin) {
        if (!ip_weights(A, bar, r0, r1)) return;
        ip_q<kIpLanes>(A, r0, r1, 0, 0.0);
        if (bar.sync()) ip_rhs<kIpLanes>(A, r0, r1, 0, 0.0);
    } else if (ip_steps(A, bar, S, r0, r1, A.dy + A.nc, 1.0)) {
        if (part == kIpMid) ip_corrector(A, bar, S, r0, r1);
        else ip_step(A, bar, S, r0, r1, 0, done + 1);
    }
}

// The SMs of the handle's device (or of the part of it that the process may use).
static int ip_blocks_resident(bchar_mesh_t m) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ip, kIpThreads, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return per_sm > 0 && sms > 0 ? sms : 1;
}

static void launch_ip(bchar_mesh_t m, const IpArgs &A, IpPart part, const IpStart &start = IpStart{}) {
    cudaMemsetAsync(&A.st->bar, 0, sizeof(unsigned), m->stream);
    if (!m->ip_resident) m->ip_resident = ip_blocks_resident(m);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(ip_grid(A.nc, m->ip_resident)));
    cfg.blockDim = dim3(kIpThreads);
    cfg.stream = m->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_ip, A, static_cast<int>(part), start);
    ++m->launches;
}

// x_e = f_e - 1 (kept in qx for the bounds / column-fix stage) and the count
// of entries within 1e-9 of a bound.
__global__ void k_ip_finish(int64_t nnz, const double *f, double *qx, DevInfo *info) {
    int at = 0;
    GRID_STRIDE(e, nnz) {
        const double fe = fmin(fmax(f[e], 0.0), 2.0);
        qx[e] = fe - 1.0;
        if (fe < 1e-9 || fe > 2.0 - 1e-9) ++at;
    }
    if (at) atomicAdd(&info->n_at_bounds, at);
}

// A solve of the conjugate gradients stops when its residual has not dropped
// by 1 % for kStallIters iterations (it cannot improve further in FP64).
constexpr int kStallIters = 400;

// The conjugate gradients with the Jacobi preconditioner (qp_precond = 0; with
// the multigrid the whole solve is one kernel, pcg.cu)
// on (A-hat D A-hat^T + diag(exc)) d = rhs, from
// d = 0 (or, with warm, from the d already in place), until z.res <= target_rz
// (z the preconditioned residual: about the squared error of d in the norm of
// the matrix, which bounds the error of A-hat^T d where the interior-point
// direction needs it -- an L1 test alone would not bound the error along the
// nearly singular modes of weakly linked cells) and max_l |res_l| / b_l <=
// target_res (after a full step, res is the constraint residual, which the
// interior point measures in that norm).  One batch of iterations is captured
// into a CUDA graph per preconditioner build (*exec; destroyed by the caller)
// and replayed until the solve has converged (its kernels do nothing then);
// the host polls once per batch.  Returns the iterations done.
static int pcg_solve(bchar_mesh_t m, const double *rhs, double target_rz, double target_res, bool warm,
                     int max_iter, cudaGraphExec_t *exec, int *graph_launches) {
    const int64_t nc = m->nc, n2 = 2 * nc;
    const int bl = blocks_for(n2);
    cudaStream_t s = m->stream;
    double *a2 = ptr<double>(m->a2), *a2c = ptr<double>(m->a2c), *diag = ptr<double>(m->diag);
    double *d = ptr<double>(m->cg_d), *res = ptr<double>(m->cg_r), *z = ptr<double>(m->cg_z);
    double *p = ptr<double>(m->cg_p), *q = ptr<double>(m->cg_q), *rp = ptr<double>(m->cg_rp);
    double *part = ptr<double>(m->partials);
    double *part_res = part + 152 * 64;
    const double *brow = ptr<double>(m->bloc), *volphi = ptr<double>(m->volphi);
    double *part_rz = part + 2 * 152 * 64;
    double *part_zp = part + 3 * 152 * 64;
    CgState *st = ptr<CgState>(m->cg);
    CgState *host_st = reinterpret_cast<CgState *>(static_cast<char *>(m->info_host.p) + sizeof(DevInfo));
    if (warm) {  // start from the d already in place: res = rhs - M d
        k_cg_reopen<<<1, 1, 0, s>>>(st);
        k_cg_matvec<<<tile_grid(2 * m->ntile), kTileThreads, kTileSmem, s>>>(
            row_view(m, a2), col_view(m, a2c), diag, d, q, part, st);
        k_residual<<<bl, kThreads, 0, s>>>(n2, rhs, q, res);
        m->launches += 3;
    } else {
        cudaMemsetAsync(d, 0, sizeof(double) * n2, s);
        k_copy<<<bl, kThreads, 0, s>>>(n2, rhs, res, nullptr);
        ++m->launches;
    }
    k_jacobi_precond<<<bl, kThreads, 0, s>>>(n2, diag, res, z, nullptr);
    k_dot<<<kRedBlocks, kThreads, 0, s>>>(n2, res, z, part_rz, nullptr);
    // the right-hand side's residual norm is not formed: the first iteration checks it
    k_cg_start<<<1, 1024, 0, s>>>(part_rz, kRedBlocks, target_rz, target_res, INFINITY, st);
    k_copy<<<bl, kThreads, 0, s>>>(n2, z, p, nullptr);
    m->launches += 4;
    const int batch = 32;
    const int mv_grid = tile_grid(2 * m->ntile);  // <= kRedBlocks partial sums of p.q
    auto enqueue_batch = [&]() {
        for (int k = 0; k < batch; ++k) {
            launch_dep_smem(k_cg_matvec, mv_grid, kTileThreads, kTileSmem, s, row_view(m, a2), col_view(m, a2c), diag, p,
                            q, part, st);
            launch_dep(k_cg_alpha, 1, 1024, s, part, mv_grid, st);
            launch_dep(k_cg_update, kRedBlocks, kThreads, s, n2, p, q, d, res, rp, brow, volphi, part_res, st);
            launch_dep(k_jacobi_precond, bl, kThreads, s, n2, diag, res, z, st);
            launch_dep(k_dot2, kRedBlocks, kThreads, s, n2, z, res, rp, part_rz, part_zp, st);
            m->launches += 5;
            launch_dep(k_cg_beta, 1, 1024, s, part_rz, part_zp, part_res, kRedBlocks, st);
            launch_dep(k_cg_pupdate, bl, kThreads, s, n2, z, p, st);
            m->launches += 2;
        }
    };
    if (!*exec) {
        const int before = m->launches;
        cudaGraph_t graph = nullptr;
        bool ok = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
        if (ok) {
            enqueue_batch();
            ok = cudaStreamEndCapture(s, &graph) == cudaSuccess && graph;
        }
        if (ok) ok = cudaGraphInstantiate(exec, graph, 0) == cudaSuccess;
        if (graph) cudaGraphDestroy(graph);
        if (!ok) {  // capture unavailable (for instance, the caller is capturing): plain launches
            cudaGetLastError();
            *exec = nullptr;
        }
        *graph_launches = m->launches - before;
        m->launches = before;
    }
    double best = INFINITY;
    int best_at = 0;
    for (;;) {
        if (*exec) {
            cudaGraphLaunch(*exec, s);
            m->launches += *graph_launches;
        } else {
            enqueue_batch();
        }
        cudaMemcpyAsync(host_st, st, sizeof(CgState), cudaMemcpyDeviceToHost, s);
        cudaStreamSynchronize(s);
        if (host_st->converged || host_st->iters >= max_iter) break;
        if (host_st->res_max < 0.99 * best) {
            best = host_st->res_max;
            best_at = host_st->iters;
        } else if (host_st->iters - best_at >= kStallIters) {
            break;
        }
    }
    return host_st->iters;
}

// Host wall clock in milliseconds (for the diagnostic trace only).
static double trace_ms() {
    timespec t;
    clock_gettime(CLOCK_MONOTONIC, &t);
    return t.tv_sec * 1e3 + t.tv_nsec * 1e-6;
}

// The elastic penalty of the constraints is quadratic up to a relative
// violation kLinearFrom and linear beyond, with slope gamma = kLinearFrom / eps^2.
constexpr double kLinearFrom = 1e-6;
// The interior-point stopping rule: scaled constraint residual <= qp_tol,
// mean complementarity <= 1e-12, the stationarity residual of 1 + x <= 1e-12 of
// the largest dual value and those of the violation parts <= 1e-12 of gamma
// (y and the multipliers reach ~gamma where the problem is infeasible, and the
// residuals then carry that much rounding).
constexpr double kIpMuTol = 1e-12;
// From here on the correctors are solved to the result's accuracy: mu falls by at most
// a factor of 1e-2 per iteration, so at least two of them are.
constexpr double kIpLastMu = 1e4 * kIpMuTol;
// The corrector's centring target never goes below kIpMuFloor: once the mean
// complementarity meets its tolerance, the iterations that are still needed to
// bring the constraint residual down hold it there instead of driving it
// towards zero (which makes the normal equations so badly conditioned that the
// inexact solves raise the constraint residual again).
constexpr double kIpMuFloor = 0.1 * kIpMuTol;
// Conjugate-gradient iterations per interior-point solve at most (the late
// normal equations are badly conditioned; an inexact direction is corrected by
// the next iteration).
constexpr int kIpCgPerSolve = 400;
constexpr double kIpRdRel = 1e-12;
constexpr double kIpStep = 0.99;
// The starting point: y = 0; the violation parts p = n = kIpStartViol with
// multipliers gamma, which satisfies their stationarity at y = 0; f = u = 1
// with multipliers kIpStartViol * gamma, so that every complementarity
// product starts equal (a centred point).  Multipliers 1 for the violation
// parts leave a dual residual of gamma = 1e8 for the first Newton step, after
// which the steps shrink to nothing on some small meshes; uncentred starts
// take up to twice the iterations on the 1024^2 workload.
constexpr double kIpStartViol = 0.1;

bchar_status launch_minimise(bchar_mesh_t m, int *cg_iters, int *ip_iters) {
    const bool trace = getenv("BCHAR_TRACE") != nullptr;  // diagnostic: per-iteration scalars on stderr
    double t_start = 0.0;
    if (trace) {
        cudaStreamSynchronize(m->stream);
        t_start = trace_ms();
    }
    const int64_t nc = m->nc, n2 = 2 * nc, nnz = m->nnz;
    const size_t zb = sizeof(double) * (nnz > 0 ? nnz : 1), nb = sizeof(double) * n2;
    Buf *ent[] = {&m->ip_f, &m->ip_u, &m->ip_zl, &m->ip_zh, &m->ip_D, &m->ip_q, &m->ip_cl, &m->ip_ch,
                  &m->ip_df, &m->ip_du, &m->ip_dzl, &m->ip_dzh};
    for (Buf *b : ent)
        if (!ensure(m, *b, zb)) return BCHAR_ERR_OUT_OF_MEMORY;
    Buf *nod[] = {&m->ip_p, &m->ip_n, &m->ip_zp, &m->ip_zn, &m->ip_cp, &m->ip_cn, &m->ip_dp, &m->ip_dn,
                  &m->ip_dzp, &m->ip_dzn};
    for (Buf *b : nod)
        if (!ensure(m, *b, nb)) return BCHAR_ERR_OUT_OF_MEMORY;
    static_assert(5 * kMaxCtas <= 4 * 152 * 64, "interior-point partials fit the scratch");
    static_assert(sizeof(CgState) + sizeof(IpScalars) <= 256, "both scalar blocks fit the cg buffer");
    cudaStream_t s = m->stream;
    const bool use_amg = m->opt.qp_precond == 1;
    const double eps2 = m->opt.penalty * m->opt.penalty;
    IpArgs A{};
    A.nc = nc;
    A.nnz = nnz;
    A.row_ptr = ptr<int64_t>(m->row_ptr);
    A.col_ptr = ptr<int64_t>(m->col_ptr);
    A.col = ptr<int32_t>(m->col);
    A.csc_src = ptr<int32_t>(m->csc_src);
    A.a = ptr<double>(m->aN);
    A.b_row = ptr<double>(m->bloc);
    A.volphi = ptr<double>(m->volphi);
    A.eps2 = eps2;
    A.gamma = kLinearFrom / eps2;
    A.pairs = 2.0 * static_cast<double>(nnz) + 2.0 * static_cast<double>(n2);
    A.mu_floor = kIpMuFloor;
    A.step = kIpStep;
    A.qp_tol = m->opt.qp_tol;
    A.mu_tol = kIpMuTol;
    A.rd_rel = kIpRdRel;
    A.max_it = m->opt.qp_max_refine;
    A.max_cg = m->opt.qp_max_iter;
    double **ent_p[] = {&A.f, &A.u, &A.zl, &A.zh, &A.D, &A.q, &A.cl, &A.ch, &A.df, &A.du, &A.dzl, &A.dzh};
    for (int k = 0; k < 12; ++k) *ent_p[k] = ptr<double>(*ent[k]);
    double **nod_p[] = {&A.p, &A.n, &A.zp, &A.zn, &A.cp, &A.cn, &A.dp, &A.dn, &A.dzp, &A.dzn};
    for (int k = 0; k < 10; ++k) *nod_p[k] = ptr<double>(*nod[k]);
    A.y = ptr<double>(m->qy);
    A.rp = ptr<double>(m->F);
    A.rhs = ptr<double>(m->rhs);
    A.dy = ptr<double>(m->cg_d);
    A.a2 = ptr<double>(m->a2);
    A.a2c = ptr<double>(m->a2c);
    A.diag = ptr<double>(m->diag);
    A.exc = ptr<double>(m->qexc);
    A.part = ptr<double>(m->partials);
    A.st = ip_scalars(m);
    // the scalars after iteration k arrive in the host's copy k % 2
    for (cudaEvent_t &e : m->ip_ev)
        if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) e = nullptr;
    unsigned char *const copies = static_cast<unsigned char *>(m->info_host.p) + sizeof(DevInfo) + sizeof(CgState);
    auto read_back = [&](int k) {
        cudaMemcpyAsync(copies + (k & 1) * kIpScalarBytes, A.st, sizeof(IpScalars), cudaMemcpyDeviceToHost, s);
        cudaEventRecord(m->ip_ev[k & 1], s);
    };
    IpScalars hs{};
    auto wait_for = [&](int k) {  // false: an error that the caller reads
        const bool ok = cudaEventSynchronize(m->ip_ev[k & 1]) == cudaSuccess && cudaPeekAtLastError() == cudaSuccess;
        memcpy(&hs, copies + (k & 1) * kIpScalarBytes, sizeof hs);
        if (ok && trace)
            fprintf(stderr, "[bchar] ip %d rp %.3e rd %.3e rpq %.3e mu %.3e dual %.3e ap %.3e ad %.3e cg %d (%.1f ms)\n",
                    hs.it, hs.rp_max, hs.rd_max, hs.rpq_max, hs.mu, hs.dual_max, hs.ap, hs.ad, hs.cg, trace_ms() - t_start);
        return ok;
    };
    // the corrector's direction is solved until its squared energy-norm error is about
    // <= 1e-2 mu (then every entry's step error stays about <= 0.1 of its distance to the
    // bound) and the constraint residual it leaves is, relative to each target, <= half
    // the current one (which the step then reduces), but not below half the stopping
    // tolerance.  The predictor's only sets the centring and the second-order terms, and
    // a thousand times looser it does that as well: 2 631 -> 1 999 CG iterations at 128^2
    // stretched, 819 -> 559 on a porous 24^3 mesh, 279 -> 139 at 32^2, with at most one to
    // three more interior-point iterations.  The corrector's system differs from the
    // predictor's only in its right-hand side: its solve starts from the predictor's direction.
    // What the last correctors leave is the result's error, so from kIpLastMu on they go
    // down to 2e-2 of the current residual and of half the tolerance (not below 1e-12, which
    // FP64 still reaches on all meshes tried).  Over 60 FP64 steps of 24^2 to 64^2 and 10^3 to 16^3 the mean
    // (geometric) relative L1 error of c against 64 bits is 3.1e-12 with 26 774 CG iterations;
    // 1.07e-11 with 25 979 without the last rule (up to 18 times more than below on uniform
    // 2D meshes), and 1.12e-11 with 75 230 when rows and columns were solved together, both
    // solves to 0.1.  A step takes about 1 % longer for it (512^2 1 074 -> 1 082 ms).
    const double half = 0.5 * m->opt.qp_tol;
    const SolveTols tols = {{1e1, 5e2, 1e3 * half}, {1e-2, 0.5, half}, {1e-2, 2e-2, fmin(half, fmax(2e-2 * half, 1e-12))},
                            kIpLastMu, kIpCgPerSolve};

    cudaMemsetAsync(A.st, 0, sizeof(IpScalars), s);
    launch_ip(m, A, kIpStart, {kIpStartViol * A.gamma, kIpStartViol, A.gamma});
    read_back(0);
    bool ok = wait_for(0), have_pattern = false;
    int total_cg = 0;
    if (ok && !hs.stop && !hs.err && use_amg) {
        if (!schur_pattern(m)) return BCHAR_ERR_OUT_OF_MEMORY;
        have_pattern = true;
        cudaMemsetAsync(m->amg.hier.p, 0, offsetof(Hier, L), s);
        if (m->amg.schur) {
            A.g = ptr<double>(m->amg.g);
            A.t = ptr<double>(m->amg.t);
        }
        // An iteration is queued before the scalars of the one before it are read, so that the
        // device does not wait for the host; the kernels of one queued in vain return at once.
        // The aggregates are found anew every other iteration (no effect on the CG iterations,
        // where every third costs up to 30 % more of them: the weights change by orders of
        // magnitude).
        int queued = 0;
        while (ok && !hs.stop && !hs.err) {
            for (; queued < hs.it + 2 && queued < A.max_it; ++queued) {
                amg_build(m, A, queued % 2 == 1);
                pcg_launch(m, A, tols);
                read_back(queued + 1);
            }
            ok = wait_for(hs.it + 1);
        }
        total_cg = hs.cg;
    }
    while (ok && !hs.stop && !hs.err && !use_amg) {
        launch_ip(m, A, kIpBegin);
        cudaGraphExec_t exec = nullptr;
        int graph_launches = 0;
        for (int corr = 0; corr < 2; ++corr) {
            const int left = m->opt.qp_max_iter - total_cg;
            const int cap = left < kIpCgPerSolve ? left : kIpCgPerSolve;
            total_cg += pcg_solve(m, A.rhs, 1e-2 * hs.mu, fmax(0.1 * hs.rp_max, half), corr == 1, cap > 0 ? cap : 1,
                                  &exec, &graph_launches);
            launch_ip(m, A, corr ? kIpEnd : kIpMid);
        }
        if (exec) cudaGraphExecDestroy(exec);
        read_back(hs.it + 1);
        ok = wait_for(hs.it + 1);
        if (total_cg >= m->opt.qp_max_iter) break;
    }
    if (hs.err) {
        m->err = "a solver kernel's grid barrier timed out";
        return BCHAR_ERR_CUDA;
    }
    const bool converged = hs.converged != 0;
    const int it = hs.it;
    k_ip_finish<<<blocks_for(nnz), kThreads, 0, s>>>(nnz, A.f, ptr<double>(m->qx), ptr<DevInfo>(m->dinfo));
    ++m->launches;
    DevInfo *di = ptr<DevInfo>(m->dinfo);
    cudaMemcpyAsync(&di->kkt_l1, &A.st->rp_max, sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (trace) {
        cudaStreamSynchronize(s);
        fprintf(stderr, "[bchar] interior point: %d iterations, %d CG iterations, %s, %.3f ms\n", it, total_cg,
                converged ? "converged" : "not converged", trace_ms() - t_start);
    }
    m->ip_iters = it;
    m->ip_converged = converged;
    *cg_iters = total_cg;
    *ip_iters = it;
    m->amg_levels = have_pattern ? hs.levels : 0;
    m->amg_coarsest = have_pattern ? hs.coarsest : 0;
    return BCHAR_OK;
}

void launch_cg_matvec_once(bchar_mesh_t m, CgState *st) {
    k_cg_matvec<<<tile_grid(2 * m->ntile), kTileThreads, kTileSmem, m->stream>>>(
        row_view(m, ptr<double>(m->a2)), col_view(m, ptr<double>(m->a2c)), ptr<double>(m->diag), ptr<double>(m->cg_p),
        ptr<double>(m->cg_q), ptr<double>(m->partials), st);
}

// ---------------------------------------------------------------- bounds, column fix, W

// a_q = a^(N) (1 + x), per row (1 + x is inside [0, 2] by construction).
__global__ void k_clip(int64_t nc, const int64_t *row_ptr, const double *aN, const double *qx, double *aq) {
    GRID_STRIDE(i, nc) {
        for (int64_t e = row_ptr[i]; e < row_ptr[i + 1]; ++e) aq[e] = aN[e] * fmin(fmax(1.0 + qx[e], 0.0), 2.0);
    }
}

// C2_j = |M_j|_phi / sum_i a_q,ij (first half of eq. volAdj).  A column whose
// entries all ended on the bound 0 keeps its A^(N) entries (dead[j] = 1).
__global__ void k_colfix(int64_t nc, const int64_t *col_ptr, const int32_t *csc_src, const double *aq,
                         const double *aN, const double *volphi, double *C2, int32_t *dead) {
    GRID_STRIDE(j, nc) {
        double s = 0.0;
        for (int64_t p = col_ptr[j]; p < col_ptr[j + 1]; ++p) s += aq[csc_src[p]];
        int d = 0;
        if (s == 0.0) {
            d = 1;
            for (int64_t p = col_ptr[j]; p < col_ptr[j + 1]; ++p) s += aN[csc_src[p]];
        }
        dead[j] = d;
        C2[j] = volphi[j] / s;
    }
}

// a_KM final, W_KM = a_KM / |K|_phi, and the relative row residual.
__global__ void k_weights(int64_t nc, const int64_t *row_ptr, const int32_t *col, const double *aq, const double *aN,
                          const int32_t *dead, const double *C2, const double *volphi, double *afin, double *wgt,
                          unsigned long long *row_res) {
    double mx = 0.0;
    GRID_STRIDE(i, nc) {
        double s = 0.0;
        const double vi = volphi[i];
        for (int64_t e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int32_t j = col[e];
            const double a = (dead[j] ? aN[e] : aq[e]) * C2[j];
            afin[e] = a;
            wgt[e] = a / vi;
            s += a;
        }
        mx = fmax(mx, fabs(s - vi) / vi);
    }
    mx = block_max(mx);
    if (threadIdx.x == 0) atomic_max_nonneg(row_res, mx);
}

void launch_finalise(bchar_mesh_t m) {
    const int64_t nc = m->nc;
    const int bl = blocks_for(nc);
    DevInfo *di = ptr<DevInfo>(m->dinfo);
    double *aq = ptr<double>(m->a2);  // reuse: a2 is no longer needed
    k_clip<<<bl, kThreads, 0, m->stream>>>(nc, ptr<int64_t>(m->row_ptr), ptr<double>(m->aN), ptr<double>(m->qx), aq);
    int32_t *dead = ptr<int32_t>(m->colfill);  // scratch: the column fill counters are no longer needed
    k_colfix<<<bl, kThreads, 0, m->stream>>>(nc, ptr<int64_t>(m->col_ptr), ptr<int32_t>(m->csc_src), aq,
                                             ptr<double>(m->aN), ptr<double>(m->volphi), ptr<double>(m->C), dead);
    k_weights<<<bl, kThreads, 0, m->stream>>>(nc, ptr<int64_t>(m->row_ptr), ptr<int32_t>(m->col), aq, ptr<double>(m->aN),
                                              dead, ptr<double>(m->C), ptr<double>(m->volphi), ptr<double>(m->afin),
                                              ptr<double>(m->wgt),
                                              reinterpret_cast<unsigned long long *>(&di->max_rel_row_res));
    k_col_error<<<bl, kThreads, 0, m->stream>>>(nc, ptr<int64_t>(m->col_ptr), ptr<int32_t>(m->csc_src),
                                                ptr<double>(m->afin), ptr<double>(m->volphi),
                                                reinterpret_cast<unsigned long long *>(&di->max_rel_col_res));
    m->launches += 4;
}

// ---------------------------------------------------------------- update (eq. phys-inter-ELLAM)

// c_out_i = sum_j W_ij c_in_j with FP64 accumulation, rounded once on store,
// tile by tile over the row view, and per-block partial sums of the three
// masses sum |K|_phi c (before, after the FP64 update, after the stored
// rounding), all in one pass.
template <class T> struct SpmvEpi {
    const double *volphi;
    const T *c_in;
    T *c_out;
    double mb, ma, ms;
    __device__ void operator()(int64_t i, double s) {
        const T stored = static_cast<T>(s);
        c_out[i] = stored;
        const double v = volphi[i];
        mb += v * static_cast<double>(c_in[i]);
        ma += v * s;
        ms += v * static_cast<double>(stored);
    }
};

template <class T>
__global__ void __launch_bounds__(kTileThreads) k_spmv(LineView V, const double *volphi, const T *c_in, T *c_out,
                                                       double *partials) {
    extern __shared__ __align__(16) unsigned char smem[];
    SpmvEpi<T> epi{volphi, c_in, c_out, 0.0, 0.0, 0.0};
    NoEpi none;
    const LineView nov{0, nullptr, nullptr, nullptr, nullptr, 0};
    tile_loop(V, c_in, epi, nov, c_in, none, smem);
    const double mb = block_sum(epi.mb);
    const double ma = block_sum(epi.ma);
    const double ms = block_sum(epi.ms);
    if (threadIdx.x == 0) {
        partials[3 * blockIdx.x] = mb;
        partials[3 * blockIdx.x + 1] = ma;
        partials[3 * blockIdx.x + 2] = ms;
    }
}

__global__ void k_mass_final(const double *partials, int n, DevInfo *info) {
    double mb = 0.0, ma = 0.0, ms = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        mb += partials[3 * i];
        ma += partials[3 * i + 1];
        ms += partials[3 * i + 2];
    }
    mb = block_sum(mb);
    ma = block_sum(ma);
    ms = block_sum(ms);
    if (threadIdx.x == 0) {
        info->mass_before = mb;
        info->mass_after = ma;
        info->mass_after_stored = ms;
    }
}

void launch_update(bchar_mesh_t m, const void *c_in, void *c_out, int c_dtype) {
    double *part = ptr<double>(m->partials);
    const int grid = tile_grid(m->ntile);
    static_assert(3 * kTileBlocks <= 4 * 152 * 64, "mass partials fit the scratch");
    const LineView V = row_view(m, ptr<double>(m->wgt));
    if (c_dtype == BCHAR_C_F32)
        k_spmv<float><<<grid, kTileThreads, kTileSmem, m->stream>>>(V, ptr<double>(m->volphi), static_cast<const float *>(c_in),
                                                            static_cast<float *>(c_out), part);
    else
        k_spmv<double><<<grid, kTileThreads, kTileSmem, m->stream>>>(V, ptr<double>(m->volphi),
                                                             static_cast<const double *>(c_in),
                                                             static_cast<double *>(c_out), part);
    k_mass_final<<<1, 1024, 0, m->stream>>>(part, grid, ptr<DevInfo>(m->dinfo));
    m->launches += 2;
}

}  // namespace bchar
