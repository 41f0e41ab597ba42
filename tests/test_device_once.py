"""Per-device set-up from several threads: whoever returns finds it done, it runs
once per device, a failure is reported and tried again.  (Contexts on different
threads share the kernels' shared memory limits; a launch that came between the
mark and the call that raises the limit was refused.)"""
import glob
import os
import subprocess

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1807_08692_gb300", "csrc")

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "hd_once.cuh"
int main() {
    HdDeviceOnce once;
    std::atomic<int> limit[2]{}, runs{0}, early{0}, bad{0};
    auto use = [&](int dev) {
        const int rc = once.run(dev, [&] {
            ++runs;
            std::this_thread::sleep_for(std::chrono::milliseconds(50));
            limit[dev] = 1;
            return 0;
        });
        if (rc) ++bad;
        if (!limit[dev]) ++early;   // a launch here would be refused
    };
    std::vector<std::thread> t;
    for (int i = 0; i < 16; ++i) t.emplace_back(use, i & 1);
    for (auto& x : t) x.join();
    HdDeviceOnce again;
    int tries = 0;
    const int first = again.run(5, [&] { ++tries; return -7; });
    const int second = again.run(5, [&] { ++tries; return 0; });
    const int third = again.run(5, [&] { ++tries; return 0; });
    std::printf("%d %d %d %d %d %d %d\n", runs.load(), early.load(), bad.load(), first, second, third, tries);
}
"""


def test_set_up_is_done_when_any_caller_returns(tmp_path):
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "once"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    assert out == ["2", "0", "0", "-7", "0", "0", "2"]


def test_every_raised_limit_goes_through_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        lines = open(path).read().split("\n")
        for i, line in enumerate(lines):
            if "cudaFuncSetAttribute(" in line:
                before = "\n".join(lines[max(0, i - 6):i])
                if "g_rank_scratch" in before:
                    continue  # hd_rank_static: its callers serialise it
                assert "HdDeviceOnce" in before and ".run(ctx->device" in before, (os.path.basename(path), i + 1)
