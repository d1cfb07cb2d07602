// A barrier across all blocks of one cooperative launch.
#pragma once

#include <cuda_runtime.h>

namespace bchar {

// A wait longer than this many clocks (about five seconds) gives up: the
// kernel records the failure and returns.
constexpr long long kSpinClocks = 10000000000LL;

// One counter in global memory, zero at launch: block arrivals add one, and
// the k-th barrier is complete when the counter reaches k times the number of
// blocks.  Thread 0's release (after the block barrier) and acquire make every
// block's earlier writes visible to all threads of every block.  About 2 350
// clocks on 16 to 152 blocks (1.2 us), against ~2.5 us for a dependent kernel
// launch; with one block it is the block barrier alone (~160 clocks).
// A grid that is one cluster (CLUSTER) has the hardware's barrier, about 450 clocks.
template <bool CLUSTER> struct GridBarT {
    static constexpr bool kCluster = CLUSTER;
    unsigned *cnt;
    int *err;
    unsigned nb, target = 0;
    __device__ GridBarT(unsigned *c, int *e, unsigned n) : cnt(c), err(e), nb(n) {}
    // false (in every thread of the block): the wait ran out, or another block's did
    __device__ bool sync() {
        if (CLUSTER && nb > 1) {
            asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
            return true;
        }
        target += nb;
        __syncthreads();
        if (nb == 1) return true;
        int ok = 1;
        if (threadIdx.x == 0) {
            unsigned v;
            // a reduction: an atomic's result would be waited for before the first poll
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
            const long long t0 = clock64();
            for (unsigned polls = 1;; ++polls) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
                if (static_cast<int>(v - target) >= 0) break;
                if ((polls & 1023u) == 0 &&
                    (clock64() - t0 > kSpinClocks || *reinterpret_cast<volatile int *>(err) != 0)) {
                    atomicExch(err, 1);
                    ok = 0;
                    break;
                }
            }
        }
        return __syncthreads_and(ok) != 0;
    }
};
using GridBar = GridBarT<false>;

// The end of a block of a cluster whose blocks read and write one another's
// shared memory and wait at the cluster's barrier.  A grid barrier that runs out
// may fail in some of its blocks and not in others (a late block completes it), and
// those go on until their next grid barrier: a failed block stays, and arrives at
// every cluster barrier, until the whole cluster has come here.  The others need one
// barrier: behind the last grid barrier nothing is exchanged.  C: done() counts
// this block among those that are here, barrier() is the cluster's, all_done()
// tells whether every block of the cluster has been counted.
template <class C> __host__ __device__ inline void leave_cluster(C &c, bool failed) {
    c.done();
    // every round but the last accompanies one barrier of another block: a few hundred at
    // most, the limit is for a block that is never counted
    for (int k = 0; k < (1 << 22); ++k) {
        c.barrier();
        if (!failed || c.all_done()) break;
    }
}

// On the device: `here` is a counter per cluster in global memory, zero at launch.
struct ClusterEnd {
    unsigned *here;
    unsigned blocks;
    __device__ void done() {
        __syncthreads();
        if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(here) : "memory");
    }
    __device__ void barrier() {
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    }
    __device__ bool all_done() {
        unsigned v = 0;
        if (threadIdx.x == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(here) : "memory");
        return __syncthreads_or(v >= blocks) != 0;
    }
};

}  // namespace bchar
