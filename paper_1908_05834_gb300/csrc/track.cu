// Tracking the balls back along the flow (Sec 2 eq. charac; Sec 3).
//
// dp/dt = sign u(p) / phi(p) is integrated by classical RK4 with `substeps`
// equal steps; sign = -1 gives F_{-dt}(p), the foot of the characteristic.
// u is the lowest-order Raviart-Thomas field of the face velocities: in cell
// c, u_a = U_a(lower face) + xi_a (U_a(upper face) - U_a(lower face)), xi_a the
// local coordinate of p in [0, 1] along axis a.
//
// A point is kept as (cell index, local coordinate) per axis rather than as an
// absolute coordinate, so that FP32 tracking keeps FP32 relative precision
// inside the cell (an absolute FP32 coordinate near 1 would only resolve 6e-8,
// about 2.5e-4 of a ball radius on a 1024^2 mesh).  A point that leaves its
// cell is moved to the neighbour ("last node <= p": a point on an interior
// face belongs to the upper cell) and is clamped to the closed box at the
// boundary.  The first stage is evaluated in the ball's own cell, so the
// points on a ball's surface that touch a face use that cell's field.
//
// The tracked radius (Sec 3): r_hat = r_K when phi is constant
// (eq. ball_volChange); otherwise the 2 d points C +- r e_a are tracked too and
// r_hat is their mean distance to the tracked centre (eq. rTrackedBall, with
// the six axis points in 3D).
#include "device.cuh"

namespace bchar {

template <class real>
__device__ __forceinline__ void relocate(const MeshView &m, int a, int &c, real &xi) {
    const real *w = Real<real>::w(m, a);
    const int n = m.n[a];
#pragma unroll 1
    for (int it = 0; it < 64; ++it) {  // one face per stage under the substep rule
        const bool up = xi >= real(1);
        if (!up && !(xi < real(0))) return;
        // one path for both directions: the lanes of a warp that leave their cells share the division
        const int cn = up ? c + 1 : c - 1;
        if (cn < 0 || cn >= n) {
            xi = up ? real(1) : real(0);
            return;
        }
        const real t = (up ? xi - real(1) : xi) * w[c] / w[cn];
        xi = up ? t : real(1) + t;
        c = cn;
    }
    xi = xi < real(0) ? real(0) : (xi > real(1) ? real(1) : xi);
}

// Arithmetic of one stage in the tracking precision.  FP64 divides by phi and
// by the width (the operations of a plain evaluation of the RT0 field); FP32
// multiplies by 1 / phi and 1 / width, all read from the cell's record (and
// formed from FP64 values).  A substep's moves and its final update use the
// width terms of the point's cell at the start of the substep, loaded once.
template <class real> struct Stage;
template <> struct Stage<double> {
    // r[0..5]: lower/upper face velocity per axis, r[6]: phi; wr[0..2]: widths
    static __device__ __forceinline__ void load(const VelView &v, int64_t k, double r[7]) {
        const double2 *p = reinterpret_cast<const double2 *>(v.recd + kRecordLen * k);
        const double2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
        r[0] = a.x, r[1] = a.y, r[2] = b.x, r[3] = b.y, r[4] = c.x, r[5] = c.y, r[6] = d.x;
    }
    static __device__ __forceinline__ void load_widths(const VelView &v, int64_t k, double wr[3]) {
        const double2 *p = reinterpret_cast<const double2 *>(v.recd + kRecordLen * k);
        const double2 e = __ldg(p + 4), f = __ldg(p + 5);
        wr[0] = e.x, wr[1] = e.y, wr[2] = f.x;
    }
    static __device__ __forceinline__ double per_phi(double u, double phi) { return u / phi; }
    // acc + u / phi
    static __device__ __forceinline__ double add_per_phi(double acc, double u, double phi) { return acc + u / phi; }
    // d over the width held in a record
    static __device__ __forceinline__ double by_width(double wr, double d) { return d / wr; }
};
template <> struct Stage<float> {
    // r[0..5]: lower/upper face velocity per axis, r[6]: 1 / phi; wr[0..2]: inverse widths
    static __device__ __forceinline__ void load(const VelView &v, int64_t k, float r[7]) {
        const float4 *p = reinterpret_cast<const float4 *>(v.recf + kRecordLen * k);
        const float4 a = __ldg(p), b = __ldg(p + 1);
        r[0] = a.x, r[1] = a.y, r[2] = a.z, r[3] = a.w, r[4] = b.x, r[5] = b.y, r[6] = b.z;
    }
    static __device__ __forceinline__ void load_widths(const VelView &v, int64_t k, float wr[3]) {
        const float4 c = __ldg(reinterpret_cast<const float4 *>(v.recf + kRecordLen * k) + 2);
        wr[0] = c.x, wr[1] = c.y, wr[2] = c.z;
    }
    static __device__ __forceinline__ float per_phi(float u, float inv_phi) { return u * inv_phi; }
    static __device__ __forceinline__ float add_per_phi(float acc, float u, float inv_phi) {
        return __fmaf_rn(u, inv_phi, acc);
    }
    // d times the inverse width held in a record (the same value as m.wif)
    static __device__ __forceinline__ float by_width(float wr, float d) { return d * wr; }
};

// Flat index of a cell (32-bit: meshes hold fewer than 2^31 cells).
template <int DIM> __device__ __forceinline__ int64_t cell_of(const MeshView &m, const int (&c)[3]) {
    return DIM == 2 ? c[0] + m.n[0] * c[1] : c[0] + m.n[0] * (c[1] + m.n[1] * c[2]);
}

// su = sign u(p) at the point (c, xi) and the record's phi term (f = sign u / phi):
// one record load.  The axis count is a template parameter so that every
// per-point array stays in registers (all loops unroll).
template <class real, int DIM>
__device__ __forceinline__ void flow(const MeshView &m, const VelView &v, const int (&c)[3], const real (&xi)[3],
                                     real sign, real (&su)[3], real &phi) {
    real r[7];
    Stage<real>::load(v, cell_of<DIM>(m, c), r);
    phi = r[6];
#pragma unroll
    for (int a = 0; a < DIM; ++a) su[a] = sign * (r[2 * a] + xi[a] * (r[2 * a + 1] - r[2 * a]));
}

// Bound by instruction issue (88 % of the slots on the porous 3D workload, FP32).
// The four stages are unrolled: as one loop body, the selects between them cost
// 12 to 16 % more time than the instruction cache gives back.  A move has one
// path for both directions with one division; with two, and all 32 lanes of a
// warp at work instead of 28, 7.1 million balls of seven points took 29.3 ms
// over 37 substeps, now 22.7.
template <class real, int DIM, int P>
__device__ __forceinline__ void rk4(const MeshView &m, const VelView &v, int (&c)[P][3], real (&xi)[P][3], real h,
                                    int substeps, real sign) {
    const real half = real(0.5) * h, sixth = h / real(6);
#pragma unroll 1
    for (int st = 0; st < substeps; ++st) {
        real acc[P][3], x2[P][3], wb[P][3];
        int c2[P][3];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            Stage<real>::load_widths(v, cell_of<DIM>(m, c[p]), wb[p]);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                c2[p][a] = c[p][a];
                x2[p][a] = xi[p][a];
                acc[p][a] = real(0);
            }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const real len = s < 2 ? half : (s == 2 ? h : sixth), wgt = s == 0 ? real(1) : real(2);
            real su[P][3], phi[P];
#pragma unroll
            for (int p = 0; p < P; ++p) flow<real, DIM>(m, v, c2[p], x2[p], sign, su[p], phi[p]);
#pragma unroll
            for (int p = 0; p < P; ++p) {
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    // the last stage moves by h/6 (k1 + 2 k2 + 2 k3 + k4), the others by their own k
                    const real k = Stage<real>::per_phi(su[p][a], phi[p]);
                    const real d = len * (s < 3 ? k : Stage<real>::add_per_phi(acc[p][a], su[p][a], phi[p]));
                    acc[p][a] = s == 0 ? k : acc[p][a] + wgt * k;
                    c2[p][a] = c[p][a];
                    x2[p][a] = xi[p][a] + Stage<real>::by_width(wb[p][a], d);
                    relocate<real>(m, a, c2[p][a], x2[p][a]);
                }
            }
        }
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                c[p][a] = c2[p][a];
                xi[p][a] = x2[p][a];
            }
    }
}

// Absolute position of (c, xi) in FP64.
template <class real>
__device__ __forceinline__ double position(const MeshView &m, int a, int c, real xi) {
    return m.x[a][c] + static_cast<double>(xi) * m.wd[a][c];
}

// Start of ball b: its cell and the local coordinate of its centre.
template <class real, int DIM>
__device__ __forceinline__ void ball_start(const MeshView &m, int64_t b, int64_t &K, int (&c0)[3], real (&xi0)[3]) {
    K = m.ball_cell[b];
    const int s = static_cast<int>(b - m.ball_off[K]);
    int cnt[3];
    unpack_counts(m.cnt[K], cnt);
    split_cell(m, K, c0);
    const int sub[3] = {s % cnt[0], (s / cnt[0]) % cnt[1], s / (cnt[0] * cnt[1])};
    xi0[0] = xi0[1] = xi0[2] = real(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) xi0[a] = (real(sub[a]) + real(0.5)) / real(cnt[a]);
}

// The balls of a block's kGroupCells consecutive cells, by their number within
// the cell and then by cell: the lanes of a warp track the same ball of
// neighbouring cells, which cross faces at the same stages.  In ball order (the
// balls of a cell side by side) the lanes diverged in almost every move, with 20
// of 32 active in the mean; with both changes 5.3 million balls take 1.27 ms over
// 20 substeps instead of 1.87.
constexpr int kGroupCells = 32;
constexpr int kListBalls = kGroupCells * kMaxBallsPerCell;  // a mesh with fuller cells is refused

struct BallList {
    int64_t first;  // first ball of the group
    int total;
    unsigned short at[kListBalls];  // list entry -> ball - first
    // every thread of the block
    __device__ void build(const MeshView &m) {
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            const int64_t K0 = static_cast<int64_t>(blockIdx.x) * kGroupCells, K = K0 + lane;
            const int64_t o0 = m.ball_off[K0];
            const int64_t o = m.ball_off[K < m.nc ? K : m.nc];
            const int n = static_cast<int>(m.ball_off[K + 1 < m.nc ? K + 1 : m.nc] - o);
            int tot = n, most = n;
            for (int d = 16; d > 0; d >>= 1) {
                tot += __shfl_xor_sync(0xffffffffu, tot, d);
                most = max(most, __shfl_xor_sync(0xffffffffu, most, d));
            }
            int base = 0;
            for (int s = 0; s < most; ++s) {
                const unsigned mask = __ballot_sync(0xffffffffu, n > s);
                const int to = base + __popc(mask & ((1u << lane) - 1u));
                if (n > s && to < kListBalls) at[to] = static_cast<unsigned short>(o - o0 + s);
                base += __popc(mask);
            }
            if (lane == 0) {
                first = o0;
                total = min(tot, kListBalls);
            }
        }
        __syncthreads();
    }
    __device__ int64_t ball(int i) const { return first + at[i]; }
};
static_assert(kGroupCells == 32, "a lane per cell");

// phi constant: r_hat = r_K, only the centres move, kBallsPerThread per lane side by side.
// By lists, a warp tracks chunks of 32 kBallsPerThread balls of its group (past its end the
// last ball again).  FP64 is bound by the FP64 pipe, which takes a warp's instruction as
// long with few lanes as with all: where the groups do not fill their chunks (stretched
// meshes, 5 balls a cell in the mean) the incomplete last ones cost it more than equal
// paths gain (1024^2 53.1 ms by lists, 45.4 without; 300^2 1.23 and 1.01; uniform 256^2,
// full chunks, 0.46 and 0.55).  There a block takes consecutive balls of the mesh, lanes four
// balls apart (cells hold four or more).  FP32: always by lists.
constexpr int kBallsPerThread = 2;
constexpr int kCentreThreads = 128;
constexpr int kCentreBalls = kCentreThreads * kBallsPerThread;  // of a block at a time

template <class real, int DIM>
__device__ __forceinline__ void track_centres(const MeshView &m, const VelView &v, real h, int substeps,
                                              const int64_t (&bs)[kBallsPerThread],
                                              const bool (&keep)[kBallsPerThread], int32_t *out_cell, real *out_xi,
                                              real *out_rhat) {
    int c[kBallsPerThread][3];
    real xi[kBallsPerThread][3];
    int64_t Ks[kBallsPerThread];
#pragma unroll
    for (int p = 0; p < kBallsPerThread; ++p) ball_start<real, DIM>(m, bs[p], Ks[p], c[p], xi[p]);
    rk4<real, DIM, kBallsPerThread>(m, v, c, xi, h, substeps, real(-1));
#pragma unroll
    for (int p = 0; p < kBallsPerThread; ++p) {
        if (!keep[p]) continue;
        const int64_t b = bs[p];
        out_cell[b] = static_cast<int32_t>(cell_of<DIM>(m, c[p]));
#pragma unroll
        for (int a = 0; a < 3; ++a) out_xi[3 * b + a] = xi[p][a];
        out_rhat[b] = Real<real>::rad(m, Ks[p]);
    }
}

template <class real, int DIM>
__global__ void __launch_bounds__(kCentreThreads, sizeof(real) == 4 ? 7 : 4)
    k_track_centres(MeshView m, VelView v, real h, int substeps, int64_t nballs, bool lists, int32_t *out_cell,
                    real *out_xi, real *out_rhat) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t bs[kBallsPerThread];
    bool keep[kBallsPerThread];
    if (sizeof(real) == 4 || lists) {
        __shared__ BallList list;
        list.build(m);
        constexpr int W = kCentreThreads / 32;
        for (int i0 = (static_cast<int>(blockIdx.y) * W + wid) * 32 * kBallsPerThread; i0 < list.total;
             i0 += static_cast<int>(gridDim.y) * W * 32 * kBallsPerThread) {
#pragma unroll
            for (int p = 0; p < kBallsPerThread; ++p) {
                const int i = i0 + p * 32 + lane;
                keep[p] = i < list.total;
                bs[p] = list.ball(keep[p] ? i : list.total - 1);
            }
            track_centres<real, DIM>(m, v, h, substeps, bs, keep, out_cell, out_xi, out_rhat);
        }
    } else {
        // two warps share 128 balls: lane l of them has 4 l .. 4 l + 3
        const int64_t base = static_cast<int64_t>(blockIdx.x) * kCentreBalls + (wid >> 1) * 128 + 4 * lane + 2 * (wid & 1);
#pragma unroll
        for (int p = 0; p < kBallsPerThread; ++p) {
            keep[p] = base + p < nballs;
            bs[p] = keep[p] ? base + p : nballs - 1;
        }
        track_centres<real, DIM>(m, v, h, substeps, bs, keep, out_cell, out_xi, out_rhat);
    }
}
static_assert(kBallsPerThread == 2 && kCentreThreads % 64 == 0, "two warps of two balls per lane share 128");

// phi varying: the centre and the 2 DIM axis points C +- r e_a are tracked;
// warp p of a block tracks point p of 32 consecutive balls (one point per lane: a
// small single-point RK4, so few registers and many warps per SM, and all lanes
// of every warp have a point), then the axis points' distances to the centres go
// through shared memory to the centres' warp, which sums them in order.  The
// points of a warp leave their cells at different stages in any order of the
// balls; in this one they read few cells' records.
template <class real, int DIM>
__global__ void __launch_bounds__(32 * (1 + 2 * DIM), (sizeof(real) == 4 ? 1400 : 900) / (32 * (1 + 2 * DIM)))
    k_track_balls(MeshView m, VelView v, real h, int substeps, int64_t nballs, int32_t *out_cell, real *out_xi,
                  real *out_rhat) {
    constexpr int G = 1 + 2 * DIM;  // points per ball
    __shared__ double cen[3][32], dist[G][32];
    const int lane = threadIdx.x & 31, p = threadIdx.x >> 5;
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * 32; i0 < nballs; i0 += static_cast<int64_t>(gridDim.x) * 32) {
        const bool valid = i0 + lane < nballs;
        const int64_t b = valid ? i0 + lane : nballs - 1;  // idle lanes track a copy and write nothing
        int64_t K;
        int c[1][3];
        real xi[1][3];
        ball_start<real, DIM>(m, b, K, c[0], xi[0]);
        {  // point p > 0: axis (p - 1) / 2, sign - for odd p, + for even p
            const real r = Real<real>::rad(m, K);
            const real sg = (p & 1) ? real(-1) : real(1);
#pragma unroll
            for (int q = 0; q < DIM; ++q)
                if (p > 0 && (p - 1) / 2 == q) xi[0][q] = xi[0][q] + sg * r / Real<real>::w(m, q)[c[0][q]];
        }
        rk4<real, DIM, 1>(m, v, c, xi, h, substeps, real(-1));
        double pos[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int q = 0; q < DIM; ++q) pos[q] = position<real>(m, q, c[0][q], xi[0][q]);
        if (p == 0)
#pragma unroll
            for (int q = 0; q < DIM; ++q) cen[q][lane] = pos[q];
        __syncthreads();
        if (p > 0) {
            double d2 = 0.0;
#pragma unroll
            for (int q = 0; q < DIM; ++q) {
                const double dq = pos[q] - cen[q][lane];
                d2 += dq * dq;
            }
            dist[p][lane] = sqrt(d2);
        }
        __syncthreads();
        if (p == 0 && valid) {
            double sum = 0.0;
#pragma unroll
            for (int q = 1; q < G; ++q) sum += dist[q][lane];
            out_cell[b] = static_cast<int32_t>(cell_of<DIM>(m, c[0]));
#pragma unroll
            for (int a = 0; a < 3; ++a) out_xi[3 * b + a] = xi[0][a];
            out_rhat[b] = static_cast<real>(sum / (2.0 * DIM));
        }
    }
}

MeshView full_view(bchar_mesh_t m);
VelView vel_view(bchar_mesh_t m);

// Every cell holds the least number of balls, and those of a group fill its chunks.
static bool full_chunks(bchar_mesh_t m) {
    const int64_t least = m->dim == 2 ? m->nb * m->nb : m->nb * m->nb * m->nb;
    return m->nballs == m->nc * least && kGroupCells * least % (32 * kBallsPerThread) == 0;
}

template <class real>
static void track_in(bchar_mesh_t m, real h, int substeps, int32_t *cell, real *xi, real *rhat) {
    MeshView mv = full_view(m);
    VelView vv = vel_view(m);
    const int64_t most = 0x7fffffff, n32 = (m->nballs + 31) / 32;
    const unsigned chunks = static_cast<unsigned>(n32 < 1 ? 1 : (n32 > most ? most : n32));
    if (m->phi_const) {
        dim3 grid(static_cast<unsigned>((m->nballs + kCentreBalls - 1) / kCentreBalls));
        const bool lists = sizeof(real) == 4 || full_chunks(m);
        if (lists) {  // a block column per group of cells, and as many blocks per group as it has chunks in the mean
            const unsigned groups = static_cast<unsigned>((m->nc + kGroupCells - 1) / kGroupCells);
            const int64_t y = ((m->nballs + groups - 1) / groups + kCentreBalls - 1) / kCentreBalls;
            grid = dim3(groups, static_cast<unsigned>(y < 1 ? 1 : (y > 64 ? 64 : y)));
        }
        if (m->dim == 2)
            k_track_centres<real, 2><<<grid, kCentreThreads, 0, m->stream>>>(mv, vv, h, substeps, m->nballs, lists, cell,
                                                                               xi, rhat);
        else
            k_track_centres<real, 3><<<grid, kCentreThreads, 0, m->stream>>>(mv, vv, h, substeps, m->nballs, lists, cell,
                                                                               xi, rhat);
    } else if (m->dim == 2) {
        k_track_balls<real, 2><<<chunks, 160, 0, m->stream>>>(mv, vv, h, substeps, m->nballs, cell,
                                                                                  xi, rhat);
    } else {
        k_track_balls<real, 3><<<chunks, 224, 0, m->stream>>>(mv, vv, h, substeps, m->nballs, cell,
                                                                                  xi, rhat);
    }
    ++m->launches;
}

void launch_track(bchar_mesh_t m, double dt, int substeps) {
    if (m->opt.precision == BCHAR_FP32_SPLIT)
        track_in<float>(m, static_cast<float>(dt / substeps), substeps, ptr<int32_t>(m->t_cell), ptr<float>(m->t_xi),
                        ptr<float>(m->t_rhat));
    else
        track_in<double>(m, dt / substeps, substeps, ptr<int32_t>(m->t_cell), ptr<double>(m->t_xi),
                         ptr<double>(m->t_rhat));
}

// Residing cells that no tracked ball reached (Sec 3.2 assumes there are
// none): the centre of such a cell M_j is carried forward over dt (F_{+dt})
// and M_j's whole porous volume is assigned to the cell K_i it lands in,
// a_ij = |M_j|_phi.  Seeds are recorded as (i << 32 | j).
template <class real, int DIM>
__global__ void k_seed_columns(MeshView m, VelView v, real h, int substeps, const int32_t *colcnt,
                               unsigned long long *seeds, DevInfo *info) {
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < m.nc;
         j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        if (colcnt[j] != 0) continue;
        int c[1][3];
        split_cell(m, j, c[0]);
        real xi[1][3] = {{real(0), real(0), real(0)}};
#pragma unroll
        for (int a = 0; a < DIM; ++a) xi[0][a] = real(0.5);
        rk4<real, DIM, 1>(m, v, c, xi, h, substeps, real(1));
        int slot = atomicAdd(&info->n_seeds, 1);
        if (slot < kMaxSeeds)
            seeds[slot] =
                (static_cast<unsigned long long>(flat_cell(m, c[0])) << 32) | static_cast<unsigned long long>(j);
        else
            atomicOr(&info->err, kErrSeeds);
    }
}

template <class real, int DIM>
static void seed_in(bchar_mesh_t m, real h, int substeps) {
    k_seed_columns<real, DIM><<<blocks_for(m->nc), kThreads, 0, m->stream>>>(
        full_view(m), vel_view(m), h, substeps, ptr<int32_t>(m->colcnt), ptr<unsigned long long>(m->seeds),
        ptr<DevInfo>(m->dinfo));
}

void launch_seed_columns(bchar_mesh_t m, double dt, int substeps) {
    const bool f32 = m->opt.precision == BCHAR_FP32_SPLIT;
    if (m->dim == 2) {
        if (f32)
            seed_in<float, 2>(m, static_cast<float>(dt / substeps), substeps);
        else
            seed_in<double, 2>(m, dt / substeps, substeps);
    } else {
        if (f32)
            seed_in<float, 3>(m, static_cast<float>(dt / substeps), substeps);
        else
            seed_in<double, 3>(m, dt / substeps, substeps);
    }
    ++m->launches;
}

// Tracked centres as absolute FP64 coordinates (for the parity tests).
template <class real>
__global__ void k_tracked_positions(MeshView m, int64_t nballs, const int32_t *t_cell, const real *t_xi,
                                    const real *t_rhat, double *pos, double *rhat) {
    for (int64_t b = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; b < nballs;
         b += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int c[3];
        split_cell(m, t_cell[b], c);
        for (int a = 0; a < 3; ++a) pos[3 * b + a] = a < m.dim ? position<real>(m, a, c[a], t_xi[3 * b + a]) : 0.0;
        rhat[b] = static_cast<double>(t_rhat[b]);
    }
}

void launch_export_tracked(bchar_mesh_t m, double *pos, double *rhat) {
    MeshView mv = full_view(m);
    if (m->opt.precision == BCHAR_FP32_SPLIT)
        k_tracked_positions<float><<<blocks_for(m->nballs), kThreads, 0, m->stream>>>(
            mv, m->nballs, ptr<int32_t>(m->t_cell), ptr<float>(m->t_xi), ptr<float>(m->t_rhat), pos, rhat);
    else
        k_tracked_positions<double><<<blocks_for(m->nballs), kThreads, 0, m->stream>>>(
            mv, m->nballs, ptr<int32_t>(m->t_cell), ptr<double>(m->t_xi), ptr<double>(m->t_rhat), pos, rhat);
    ++m->launches;
}

}  // namespace bchar
