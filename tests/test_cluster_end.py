"""A block whose grid barrier ran out must not leave its cluster while the other
blocks may still reach into its shared memory or wait for it at the cluster's
barrier.  The protocol of gridbar.cuh is run here on host threads, one per
block: a cluster barrier that counts out those that have exited (as the
hardware's does), memory that is gone with its block, and a grid barrier that
fails in chosen blocks while the others pass it.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_05834_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>
#include "gridbar.cuh"

constexpr int kBlocks = 8, kRounds = 4, kExchanges = 5;

struct Barrier {  // of the threads that have not exited
    std::mutex m;
    std::condition_variable cv;
    int members = kBlocks, waiting = 0;
    long phase = 0;
    void open() {
        waiting = 0;
        ++phase;
        cv.notify_all();
    }
    void wait() {
        std::unique_lock<std::mutex> l(m);
        const long p = phase;
        if (++waiting == members) open();
        else cv.wait(l, [&] { return phase != p; });
    }
    void exit() {
        std::unique_lock<std::mutex> l(m);
        if (--members > 0 && waiting == members) open();
    }
};

struct Cluster {
    Barrier bar;
    std::atomic<int> here{0}, alive[kBlocks], bad{0};
};
struct End {
    Cluster &c;
    void done() { c.here.fetch_add(1); }
    void barrier() { c.bar.wait(); }
    bool all_done() { return c.here.load() >= kBlocks; }
};

// Block b's grid barrier of round r fails when it is one of `late` (bits) in the
// round `at`; from the next round on it fails in all blocks.
static void block(Cluster &c, int b, int at, unsigned late) {
    bool go = true;
    for (int r = 0; r < kRounds && go; ++r) {
        go = r < at || (r == at && !((late >> b) & 1));
        if (!go) break;
        for (int k = 0; k < kExchanges; ++k) {
            for (int q = 0; q < kBlocks; ++q)
                if (!c.alive[q].load()) c.bad.fetch_add(1);
            c.bar.wait();
        }
    }
    End end{c};
    bchar::leave_cluster(end, !go);
    c.alive[b].store(0);
    c.bar.exit();
}

int main() {
    int bad = 0;
    for (int at = 0; at <= kRounds; ++at)
        for (unsigned late = 0; late < (1u << kBlocks); late += at < kRounds ? 3 : 1u << kBlocks) {
            Cluster c;
            for (auto &a : c.alive) a.store(1);
            std::vector<std::thread> t;
            for (int b = 0; b < kBlocks; ++b) t.emplace_back(block, std::ref(c), b, at, late);
            for (auto &x : t) x.join();
            bad += c.bad.load();
        }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which(os.environ.get("NVCC", "nvcc")) is None, reason="needs nvcc (host code only)")
def test_a_failed_block_stays_until_its_cluster_is_done(tmp_path):
    src, exe = tmp_path / "end.cu", tmp_path / "end"
    src.write_text(PROGRAM)
    r = subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-O1", "-arch=sm_103a",
                        "-I", CSRC, "-o", str(exe), str(src), "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, f"{r.stdout.strip()} accesses to the memory of a block that had left"
