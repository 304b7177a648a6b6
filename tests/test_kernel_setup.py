"""The opt-ins to shared memory: one per kernel and device, never taken back
by a smaller one, whichever threads launch (compiled for the host with a fake
of the call that sets the attribute)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2601_11808_gb300", "csrc")

MAIN = r"""
#include "kernel_setup.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

int main()
{
    sivf::KernelSetup su;
    std::atomic<size_t> value[2];          // the attribute on two devices
    std::atomic<int> calls[2], bad{0};
    for (int d = 0; d < 2; ++d) value[d] = 48, calls[d] = 0;
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 20000; ++i) {
                const int d = (t + i) & 1;
                const size_t smem = 40 + (size_t)((i / 2 * 7 + t * 13) % 180);
                su.opt_in(d, smem, 48, [&](size_t n) { value[d] = n; ++calls[d]; return true; });
                if (smem > value[d]) ++bad;    // the launch would fail
                if (su.resident(d, smem, [&] { return (int)smem * 2 + d; }) != (int)smem * 2 + d) ++bad;
            }
        });
    for (auto &t : ts) t.join();
    for (int d = 0; d < 2; ++d) if (value[d] != 219 || calls[d] < 1 || calls[d] > 180) ++bad;
    // one that failed is asked for again
    int tries = 0;
    su.opt_in(2, 100, 48, [&](size_t) { ++tries; return false; });
    su.opt_in(2, 100, 48, [&](size_t) { ++tries; return true; });
    su.opt_in(2, 90, 48, [&](size_t) { ++tries; return true; });
    if (tries != 2) ++bad;
    printf("%d\n", (int)bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_opt_ins_of_devices_and_threads(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True, timeout=120)


def test_no_opt_in_is_kept_per_process():
    """Every opt-in goes through the one that knows the device."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            assert "cudaFuncSetAttribute(" not in open(os.path.join(CSRC, f)).read(), f
