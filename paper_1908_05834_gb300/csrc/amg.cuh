// Declarations of the linear solver of the minimisation: the column pattern of
// the row-eliminated normal equations (schur.cu), the aggregation-multigrid
// hierarchy (amg.cu) and the preconditioned conjugate gradients (pcg.cu).
#pragma once

#include "internal.cuh"

namespace bchar {

constexpr int kMaxLevels = 40;
constexpr int kMaxCtas = 256;        // blocks of the cooperative kernels at most
constexpr int kWideCluster = 8;      // blocks per cluster of a solve across the grid
constexpr int kSmallCluster = 16;    // of a solve by one cluster alone
constexpr int kSolveThreads = 512;   // threads per block of the conjugate gradients
constexpr int kBuildThreads = 1024;  // threads per block of the hierarchy build
constexpr int kDense = 32;           // a coarsest level of at most this many nodes is solved by its inverse

// Levels of at most this many off-diagonal entries and nodes are built by block 0
// alone, between block barriers.  (At 4 000 the first such level took it 33 us for
// the values and 52 in full, against 9 and 35 for a level across the grid.)
constexpr int kBlockEntries = 1200;
constexpr int kBlockNodes = 1500;
constexpr int kBlockTotalNodes = 2600;  // nodes of all such levels at most

// Where one block's share of a level is: its rows (the members of its
// aggregates, in aggregate order, then its nodes without a coarse counterpart)
// in the level's order array, and its aggregates.
struct Seg {
    int m0, mlen, l0, llen, g0, glen;
};

struct LevelInfo {
    int64_t noff;   // first node of the level in the node arrays
    int64_t nnz;    // off-diagonal entries
    int n;          // nodes
    int nmem;       // nodes that have a coarse counterpart
    int grid;       // 1: shared by all blocks, 0: block 0 alone
};

// Control block of the hierarchy and the solves.
struct Hier {
    unsigned bar[3];          // barrier counters: build (zeroed by the solves), solves (by the build), stage timing
    int notier[2];            // (solves, stage timing) the first cluster's levels do not fit its shared memory
    unsigned left[2][kMaxCtas / kWideCluster];  // (solves, stage timing) blocks at their end, per cluster (zeroed by the build)
    int general;              // a block's rows of the finest level do not fit its shared memory (zeroed by the build)
    // set by a build with new aggregates
    int overflow;             // the entry arrays are full: coarsening stops
    unsigned long long ecur;  // entries in use
    unsigned mcur[kMaxLevels];
    unsigned long long nnzacc[kMaxLevels];
    int nlev;
    int dense;   // the coarsest level is solved by its inverse
    int sweeps;  // else by this many Jacobi sweeps (even)
    LevelInfo L[kMaxLevels];
    int ctasum[2][kMaxCtas];
    double part[4][kMaxCtas];
    double inv[kDense * kDense];
};

// The level arrays (device pointers), passed by value to the kernels.
struct HierView {
    Hier *H;
    Seg *seg;  // kMaxLevels x kMaxCtas
    int64_t capn, cape;
    int64_t *rs;                    // first entry of each row
    int32_t *rl;                    // entries of each row
    double *dg, *ex, *om, *x, *b;   // diagonal, excess, smoother weight, V-cycle vectors
    int32_t *own;                   // a level's nodes grouped by aggregate, then those without a coarse counterpart
    int32_t *gs, *gc;               // per coarse node: first member in the finer level's own, members
    int32_t *agg, *raw;             // aggregate of each node (-1: none); entries of a coarse node's members
    int32_t *ecol;
    double *ew;                     // weights w > 0: the operator is diag - W
};

// Shape of the cooperative kernels for the current finest level.
struct SolveShape {
    int grid, cluster, small;
};
struct IpArgs;  // ip.cuh
// The clusters of a kernel that the current device holds at once (false: it refuses the shape).
template <class K> inline bool clusters_resident(K kernel, int cluster, int threads, size_t smem, int *n) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(n, kernel, &cfg) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}
// What a device holds at once of the solve and build kernels.
struct SolveRoom {
    int blocks = 0;       // of clusters of kWideCluster, one block per SM (0: not asked yet)
    bool small = false;   // one cluster of kSmallCluster
};
void pcg_opt_in();  // before the first launch on a device, like tiles_opt_in
void amg_opt_in();
SolveRoom solve_room();  // pcg.cu (asks the device)
bool build_cluster_fits();  // amg.cu: one cluster of kSmallCluster of the build
SolveShape solve_shape(bchar_mesh_t m);

// A finest level of at most this size is solved by one cluster: a pass of its
// kSmallCluster blocks takes about 1 300 clocks plus 19 per FP64 warp instruction
// (0.06 clocks per entry), one across the grid about 4 000.  Three more clusters
// that share the passes over A's entries took 3 % off a 64^2 step alone, but a
// batch of seven small meshes took 58 ms instead of 36: their launches no longer
// fit side by side.
constexpr int64_t kSmallEntries = 40000;
constexpr int64_t kSmallNodes = 4096;

// Dynamic shared memory of a block of the solve kernel.  From kLargeEntries entries of
// the finest level per block on (192 KB of columns and weights alone) its rows are read
// from global memory, and the shared memory that is not asked for is L1: with 20 KB of
// it, the sectors of the rows that a block's warps walk side by side were evicted and
// fetched several times.  A step with 200 KB and with 128 to 144 KB, in ms: porous 48^3 (22 000
// entries a block) 792 and 620, 64^3 3 350 and 1 890, 96^3 20 200 and 9 110, 128^3 49 000 and
// 26 000, 1024^2 (45 000) 6 640 and 5 370; below the line 40^3 (10 600) 354 and 392,
// 256^2 (2 600) 295 and 335, 448^2 (8 200) 856 and 878, 512^2 (10 800) 1 074 and 1 039.
// With 112 KB the first cluster's levels do not always fit (96^3: 3 950 -> 5 020 iterations).
constexpr size_t kSolveSmem = 200 * 1024, kLargeSmem = 144 * 1024;
constexpr int64_t kLargeEntries = 16000;
inline size_t solve_smem_of(int64_t e0, int blocks) { return e0 > kLargeEntries * blocks ? kLargeSmem : kSolveSmem; }

inline SolveShape solve_shape_of(int64_t e0, int64_t n0, const SolveRoom &room) {
    if (room.small && e0 <= kSmallEntries && n0 <= kSmallNodes) return {kSmallCluster, kSmallCluster, 1};
    // one block per ~300 entries (two warps of rows), as many as the device holds
    int64_t g = (e0 / 300 + kWideCluster - 1) / kWideCluster * kWideCluster;
    if (g < 2 * kWideCluster) g = 2 * kWideCluster;
    const int most = kMaxCtas / kWideCluster * kWideCluster;
    if (g > most) g = most;
    if (g > room.blocks) g = room.blocks;
    return {static_cast<int>(g), kWideCluster, 0};
}

// The limits of the system with the rows eliminated, per entry of A (schur.cu): the
// contributions (pairs of entries of one row of A), and its entries.  At 12 pairs it
// holds about five entries per entry of A where the product through the two views
// touches two (measured 4.1 to 5.3 between 9 and 17 pairs); the recipes' matrices have
// 2 to 5.  The second limit only bounds the memory.
constexpr int64_t kMaxPairs = 12, kMaxFill = 6;
// Room in the level arrays: all levels together, of the finest level's nodes and entries.
constexpr int64_t kRoomNodes10 = 26, kRoomEntries = 4;

// Bytes per cell of schur_pattern's buffers, at most, where A's rows hold `rows` entries
// in the mean and an entry of A costs per_entry bytes besides: the larger of the two
// forms, as the difference to per_entry * rows.  Buffers have an eighth to spare.
inline double solver_bytes_per_cell(double rows, double per_entry) {
    // per node: rs, three or five arrays of each type (72 bytes), eight of the matching's, seven vectors
    const double node = 1.125 * (72.0 * kRoomNodes10 / 10 + 8 * 4 + 7 * 8);
    const double cell = 8 + 4 + 8, entry = 1.125 * 8;  // t, counts and offsets of the contributions; g
    const double both = 2 * node + cell + rows * (entry + 1.125 * 12 * kRoomEntries * 2);
    // at most kMaxPairs contributions per entry: the squares of the row lengths sum to at most
    // (kMaxPairs + 1) times their sum, so a row has at most kMaxPairs + 1 entries in the mean
    const double r = rows < kMaxPairs + 1 ? rows : kMaxPairs + 1;
    const double eliminated = node + cell + r * (entry + 1.125 * (12 * kMaxPairs + (12 * kRoomEntries + 4) * kMaxFill));
    const double e = eliminated - per_entry * (rows - r);
    return both > e ? both : e;
}

// Once per step: the finest level's pattern (false: out of memory).
bool schur_pattern(bchar_mesh_t m);
// An interior-point iteration: the weights of the normal equations and the
// hierarchy for them; with same_aggregates the values alone, on the aggregates
// of the build before.
void amg_build(bchar_mesh_t m, const IpArgs &ip, bool same_aggregates);
// Its predictor and corrector, the step and the residuals after it.  A solve stops at
// z.res <= rz_rel mu, max |res_l| / b_l <= max(res_rel rp_max, res_floor).
struct SolveTol {
    double rz_rel, res_rel, res_floor;
};
struct SolveTols {
    SolveTol predictor, corrector, last;  // last: the corrector's once mu <= last_mu
    double last_mu;
    int max_iter;   // of one solve
};
void pcg_launch(bchar_mesh_t m, const IpArgs &ip, const SolveTols &tols);
void amg_release(Amg &amg);
HierView hier_view(bchar_mesh_t m);
// Timing aids: one damped-Jacobi sweep of the finest level; one V-cycle.
void amg_smooth_once(bchar_mesh_t m);
void amg_vcycle_once(bchar_mesh_t m);

}  // namespace bchar
