"""The shared memory opt-in of a kernel that several threads launch with different
sizes (smem_opt_in.h): never below what any of them has been told it may use."""
import os
import subprocess

from tests.libutil import ROOT

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "smem_opt_in.h"

int main() {
    for (int round = 0; round < 30; ++round) {
        SmemOptIn state;
        std::atomic<size_t> attribute[2] = {{48 * 1024}, {48 * 1024}};   // as the runtime keeps it: the last call wins
        std::atomic<int> low{0}, carves{0}, waiting{0};
        std::vector<std::thread> threads;
        for (int t = 0; t < 8; ++t)
            threads.emplace_back([&, t] {
                for (++waiting; waiting < 8;) std::this_thread::yield();   // all at once
                for (int i = 0; i < 6; ++i) {
                    const int dev = t & 1;
                    const size_t smem = 1024 * (40 + 16 * ((t * 5 + i * 3) % 8));
                    state.require(
                        dev, smem, true,
                        [&](size_t n) {
                            std::this_thread::sleep_for(std::chrono::microseconds(37 * ((t + i) % 5)));
                            attribute[dev] = n;
                        },
                        [&] { ++carves; });
                    if (attribute[dev] < smem) ++low;   // this thread's launch would be refused
                }
            });
        for (auto& t : threads) t.join();
        if (low || carves != 2) return 1;
        state.require(-1, 200 * 1024, false, [&](size_t n) { attribute[0] = n; }, [] {});   // a device beyond the table
        if (attribute[0] != 200 * 1024) return 2;
    }
    return 0;
}
"""


def test_threads_never_lower_the_opt_in(tmp_path):
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "main")
    csrc = os.path.join(ROOT, "paper_2505_15771_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + csrc, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_kernels_opt_in_through_it():
    csrc = os.path.join(ROOT, "paper_2505_15771_gb300", "csrc")
    for f in ("stage_kernels.cuh", "stage_tc.cu", "sdirk_bj.cu", "stage_team.cuh", "stage.cu"):
        src = open(os.path.join(csrc, f)).read()
        assert src.count("cudaFuncAttributeMaxDynamicSharedMemorySize") == (1 if f == "stage_kernels.cuh" else 0), f
