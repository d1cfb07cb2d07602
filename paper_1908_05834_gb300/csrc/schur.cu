// The finest level of the minimisation's linear system, once per step.
//
// The normal equations couple row nodes only to column nodes, so the rows are
// eliminated exactly: the system on the columns is again an M-matrix,
//   S_jk = -sum_i w_ij w_ik / D_i,   shift_j = exc_j + sum_i w_ij exc_i / D_i
// (w = a^2 D the weights, D_i the diagonal of row i, exc the shifts: sums of
// positive terms, nothing cancels).  Half the unknowns, one level less, and
// the conjugate gradients need fewer iterations (128^2 stretched: 3 035 on
// rows and columns, 2 545 on the columns; porous 24^3: 1 016 and 810).
//
// The pattern depends on A alone, so it is formed once per step, with the
// contributions of every entry (pairs of entries of one row of A) in a fixed
// order; each interior-point iteration then only sums products (amg.cu).  A
// matrix whose rows are so long that the products would outweigh the gain
// (more than kMaxPairs contributions or kMaxFill entries per entry of A), or where
// one column collects more than kBlockPairs, keeps rows and columns as they are.
#include "amg.cuh"
#include "device.cuh"

namespace bchar {

constexpr int kWarpPairs = 512;    // contributions of a column sorted by one warp
constexpr int kBlockPairs = 8192;  // by one block
static_assert(kWarpPairs >= 32 && (kWarpPairs & (kWarpPairs - 1)) == 0 && (kBlockPairs & (kBlockPairs - 1)) == 0,
              "the sorts pad to a power of two of at least 32");
constexpr size_t kBlockPairSmem = static_cast<size_t>(kBlockPairs) * (sizeof(unsigned long long) + sizeof(int2));

struct PairStat {
    unsigned long long total;
    int most;
};

__global__ void k_pair_counts(int64_t nc, const int64_t *row_ptr, const int64_t *col_ptr, const int32_t *csc_row,
                              int32_t *cnt, PairStat *st) {
    int most = 0;
    unsigned long long tot = 0;
    for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < nc;
         j += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int64_t r = 0;
        for (int64_t p = col_ptr[j]; p < col_ptr[j + 1]; ++p) {
            const int32_t i = csc_row[p];
            r += row_ptr[i + 1] - row_ptr[i] - 1;
        }
        const int c = r > 0x3fffffff ? 0x3fffffff : static_cast<int>(r);
        cnt[j] = c;
        most = max(most, c);
        tot += static_cast<unsigned long long>(r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&st->most, most);
        atomicAdd(&st->total, tot);
    }
}

// Gathers the contributions of column j (one warp): keys (other column << 32 |
// arrival) and the two entries of A; rows in increasing order.
__device__ int gather_pairs(int64_t j, const int64_t *row_ptr, const int32_t *col, const int64_t *col_ptr,
                            const int32_t *csc_row, const int32_t *csc_src, unsigned long long *keys, int2 *pairs) {
    const int lane = threadIdx.x & 31;
    int n = 0;
    for (int64_t p = col_ptr[j]; p < col_ptr[j + 1]; ++p) {
        const int32_t i = csc_row[p], e1 = csc_src[p];
        const int64_t b = row_ptr[i], e = row_ptr[i + 1];
        for (int64_t base = b; base < e; base += 32) {
            const int64_t k = base + lane;
            const int32_t c = k < e ? col[k] : static_cast<int32_t>(j);
            const bool keep = c != j;
            const unsigned mask = __ballot_sync(0xffffffffu, keep);
            const int at = n + __popc(mask & ((1u << lane) - 1u));
            if (keep) {
                keys[at] = (static_cast<unsigned long long>(static_cast<unsigned>(c)) << 32) | static_cast<unsigned>(at);
                pairs[at] = make_int2(e1, static_cast<int>(k));
            }
            n += __popc(mask);
        }
    }
    return n;
}

template <class Sync>
__device__ void sort_pairs(unsigned long long *keys, int n, int tid, int nt, Sync sync) {
    int P = 32;
    while (P < n) P <<= 1;
    for (int i = n + tid; i < P; i += nt) keys[i] = ~0ull;
    sync();
    for (int k = 2; k <= P; k <<= 1)
        for (int s = k >> 1; s > 0; s >>= 1) {
            for (int i = tid; i < P; i += nt) {
                const int l = i ^ s;
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

// Writes column j's contributions in key order and returns its distinct
// columns (one warp, after the sort).
__device__ int put_pairs(int64_t off, int n, const unsigned long long *keys, const int2 *pairs, int32_t *raw_key,
                         int2 *raw_pair) {
    const int lane = threadIdx.x & 31;
    int runs = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        bool start = false;
        if (i < n) {
            const unsigned long long k = keys[i];
            raw_key[off + i] = static_cast<int32_t>(k >> 32);
            raw_pair[off + i] = pairs[k & 0xffffffffull];
            start = i == 0 || (keys[i - 1] >> 32) != (k >> 32);
        }
        runs += __popc(__ballot_sync(0xffffffffu, start));
    }
    return runs;
}

__global__ void __launch_bounds__(128) k_schur_columns(int64_t nc, const int64_t *row_ptr, const int32_t *col,
                                                       const int64_t *col_ptr, const int32_t *csc_row,
                                                       const int32_t *csc_src, const int32_t *cnt, const int64_t *off,
                                                       int32_t *raw_key, int2 *raw_pair, int32_t *rl) {
    __shared__ unsigned long long keys_all[4][kWarpPairs];
    __shared__ int2 pairs_all[4][kWarpPairs];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long *keys = keys_all[wid];
    int2 *pairs = pairs_all[wid];
    for (int64_t j = blockIdx.x * 4ll + wid; j < nc; j += gridDim.x * 4ll) {
        const int c = cnt[j];
        if (c > kWarpPairs) continue;  // warp-uniform
        const int n = gather_pairs(j, row_ptr, col, col_ptr, csc_row, csc_src, keys, pairs);
        __syncwarp();
        sort_pairs(keys, n, lane, 32, [] { __syncwarp(); });
        const int runs = put_pairs(off[j], n, keys, pairs, raw_key, raw_pair);
        if (lane == 0) rl[j] = runs;
        __syncwarp();
    }
}

// The columns with more than kWarpPairs contributions, one block each.
__global__ void __launch_bounds__(1024) k_schur_wide(int64_t nc, const int64_t *row_ptr, const int32_t *col,
                                                     const int64_t *col_ptr, const int32_t *csc_row,
                                                     const int32_t *csc_src, const int32_t *cnt, const int64_t *off,
                                                     int32_t *raw_key, int2 *raw_pair, int32_t *rl) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(smem);
    int2 *pairs = reinterpret_cast<int2 *>(smem + sizeof(unsigned long long) * kBlockPairs);
    for (int64_t j = blockIdx.x; j < nc; j += gridDim.x) {
        const int c = cnt[j];
        if (c <= kWarpPairs || c > kBlockPairs) continue;  // block-uniform
        if (threadIdx.x < 32) gather_pairs(j, row_ptr, col, col_ptr, csc_row, csc_src, keys, pairs);
        __syncthreads();
        sort_pairs(keys, c, threadIdx.x, blockDim.x, [] { __syncthreads(); });
        if (threadIdx.x < 32) {
            const int runs = put_pairs(off[j], c, keys, pairs, raw_key, raw_pair);
            if (threadIdx.x == 0) rl[j] = runs;
        }
        __syncthreads();
    }
}

// The entries: their column and their first contribution.
__global__ void k_schur_entries(int64_t nc, const int32_t *cnt, const int64_t *off, const int32_t *raw_key,
                                const int64_t *rs, int32_t *ecol, uint32_t *cs) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t j = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; j < nc; j += nw) {
        const int n = cnt[j];
        const int64_t o = off[j], dst = rs[j];
        int runs = 0;
        for (int base = 0; base < n; base += 32) {
            const int i = base + lane;
            const int32_t k = i < n ? raw_key[o + i] : -1;
            const bool start = i < n && (i == 0 || raw_key[o + i - 1] != k);
            const unsigned mask = __ballot_sync(0xffffffffu, start);
            if (start) {
                const int64_t at = dst + runs + __popc(mask & ((1u << lane) - 1u));
                ecol[at] = k;
                cs[at] = static_cast<uint32_t>(o + i);
            }
            runs += __popc(mask);
        }
        if (j == nc - 1 && lane == 0) cs[dst + runs] = static_cast<uint32_t>(o + n);
    }
}

// Rows and columns: row node l < n_c holds row l (columns as n_c + j), node
// n_c + j column j.
__global__ void k_bipartite_rows(int64_t nc, int64_t nnz, const int64_t *row_ptr, const int32_t *col,
                                 const int64_t *col_ptr, const int32_t *csc_row, int64_t *rs, int32_t *rl,
                                 int32_t *ecol) {
    for (int64_t l = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; l < 2 * nc;
         l += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const bool row = l < nc;
        const int64_t b = row ? row_ptr[l] : col_ptr[l - nc], e = row ? row_ptr[l + 1] : col_ptr[l - nc + 1];
        const int64_t dst = row ? b : nnz + b;
        rs[l] = dst;
        rl[l] = static_cast<int32_t>(e - b);
        for (int64_t k = b; k < e; ++k) ecol[dst + k - b] = row ? static_cast<int32_t>(nc + col[k]) : csc_row[k];
    }
}

// A buffer with an eighth to spare, so that the next steps' slightly larger
// matrices do not reallocate it.
static bool ensure_more(bchar_mesh_t m, Buf &b, size_t bytes) {
    return (b.p && b.bytes >= bytes) || ensure(m, b, bytes + bytes / 8) || ensure(m, b, bytes);
}

// The arrays of a system of n0 nodes, its hierarchy and its conjugate gradients.
static bool node_buffers(bchar_mesh_t m, int64_t n0) {
    Amg &A = m->amg;
    A.n0 = n0;
    A.capn = n0 * kRoomNodes10 / 10 + 256;
    const size_t cn = static_cast<size_t>(A.capn);
    for (Buf *b : {&A.dg, &A.ex, &A.om, &A.x, &A.b})
        if (!ensure_more(m, *b, sizeof(double) * cn)) return false;
    for (Buf *b : {&A.rl, &A.own, &A.gs, &A.gc, &A.agg, &A.raw})
        if (!ensure_more(m, *b, sizeof(int32_t) * cn)) return false;
    return ensure_more(m, A.rs, sizeof(int64_t) * cn) && ensure_more(m, A.scratch, sizeof(int32_t) * 8 * n0) &&
           ensure_more(m, A.vec, sizeof(double) * 7 * n0);
}

static bool entry_buffers(bchar_mesh_t m, int64_t e0) {
    Amg &A = m->amg;
    A.e0 = e0;
    A.cape = kRoomEntries * e0 + 4096;
    return ensure_more(m, A.ecol, sizeof(int32_t) * A.cape) && ensure_more(m, A.ew, sizeof(double) * A.cape);
}

// The system with the rows eliminated; A.schur is false on return when it has more
// than kMaxFill entries per entry of A.  False: out of memory.
static bool eliminated_form(bchar_mesh_t m, const PairStat &h) {
    Amg &A = m->amg;
    cudaStream_t s = m->stream;
    const int64_t nc = m->nc;
    const int64_t *row_ptr = ptr<int64_t>(m->row_ptr), *col_ptr = ptr<int64_t>(m->col_ptr);
    const int32_t *col = ptr<int32_t>(m->col), *csc_row = ptr<int32_t>(m->csc_row), *csc_src = ptr<int32_t>(m->csc_src);
    const size_t tot = h.total > 0 ? static_cast<size_t>(h.total) : 1;
    if (!node_buffers(m, nc) || !ensure_more(m, A.raw_key, sizeof(int32_t) * tot) ||
        !ensure_more(m, A.pair, sizeof(int2) * tot))
        return false;
    int32_t *cnt = ptr<int32_t>(A.raw_cnt), *key = ptr<int32_t>(A.raw_key), *rl = ptr<int32_t>(A.rl);
    int64_t *off = ptr<int64_t>(A.raw_off), *rs = ptr<int64_t>(A.rs);
    scan_i32_to_i64(m, cnt, off, nc);
    k_schur_columns<<<blocks_for(nc * 32, 128), 128, 0, s>>>(nc, row_ptr, col, col_ptr, csc_row, csc_src, cnt, off, key,
                                                             ptr<int2>(A.pair), rl);
    ++m->launches;
    if (h.most > kWarpPairs) {
        cudaFuncSetAttribute(k_schur_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBlockPairSmem));
        k_schur_wide<<<static_cast<int>(nc < 152 ? nc : 152), 1024, kBlockPairSmem, s>>>(
            nc, row_ptr, col, col_ptr, csc_row, csc_src, cnt, off, key, ptr<int2>(A.pair), rl);
        ++m->launches;
    }
    scan_i32_to_i64(m, rl, rs, nc);
    int64_t e0 = 0;
    cudaMemcpyAsync(&e0, rs + nc, sizeof e0, cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) return true;  // the caller reads the error
    A.schur = e0 <= kMaxFill * m->nnz;
    if (!A.schur) return true;
    if (!entry_buffers(m, e0) || !ensure_more(m, A.cs, sizeof(uint32_t) * (e0 + 1))) return false;
    k_schur_entries<<<blocks_for(nc * 32), kThreads, 0, s>>>(nc, cnt, off, key, rs, ptr<int32_t>(A.ecol), ptr<uint32_t>(A.cs));
    ++m->launches;
    return true;
}

static bool bipartite_form(bchar_mesh_t m) {
    Amg &A = m->amg;
    for (Buf *b : {&A.raw_key, &A.pair, &A.cs}) release(*b);  // of an eliminated system before
    if (!node_buffers(m, 2 * m->nc) || !entry_buffers(m, 2 * m->nnz)) return false;
    k_bipartite_rows<<<blocks_for(2 * m->nc), kThreads, 0, m->stream>>>(
        m->nc, m->nnz, ptr<int64_t>(m->row_ptr), ptr<int32_t>(m->col), ptr<int64_t>(m->col_ptr), ptr<int32_t>(m->csc_row),
        ptr<int64_t>(A.rs), ptr<int32_t>(A.rl), ptr<int32_t>(A.ecol));
    ++m->launches;
    return true;
}

bool schur_pattern(bchar_mesh_t m) {
    Amg &A = m->amg;
    cudaStream_t s = m->stream;
    const int64_t nc = m->nc, nnz = m->nnz;
    if (!ensure(m, A.hier, sizeof(Hier)) || !ensure(m, A.seg, sizeof(Seg) * kMaxLevels * kMaxCtas) ||
        !ensure(m, A.stat, sizeof(PairStat)) || !ensure(m, A.raw_cnt, sizeof(int32_t) * nc) ||
        !ensure(m, A.raw_off, sizeof(int64_t) * (nc + 1)) || !ensure(m, A.t, sizeof(double) * nc) ||
        !ensure_more(m, A.g, sizeof(double) * (nnz > 0 ? nnz : 1)))
        return false;
    PairStat *st = ptr<PairStat>(A.stat);
    cudaMemsetAsync(st, 0, sizeof(PairStat), s);
    k_pair_counts<<<blocks_for(nc), kThreads, 0, s>>>(nc, ptr<int64_t>(m->row_ptr), ptr<int64_t>(m->col_ptr),
                                                      ptr<int32_t>(m->csc_row), ptr<int32_t>(A.raw_cnt), st);
    ++m->launches;
    PairStat h{};
    cudaMemcpyAsync(&h, st, sizeof h, cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) return true;  // the caller reads the error
    A.schur = h.most <= kBlockPairs && h.total <= static_cast<unsigned long long>(kMaxPairs * nnz) &&
              h.total < 0xffffffffull;
    if (A.schur && !eliminated_form(m, h)) {
        // no room for it: at ten entries per row it takes twice what rows and columns do
        for (Buf *b : {&A.raw_key, &A.pair, &A.cs, &A.ecol, &A.ew}) release(*b);
        A.schur = false;
        m->err.clear();
    }
    return A.schur || bipartite_form(m);
}

}  // namespace bchar
