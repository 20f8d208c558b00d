"""Set-up that is kept per device (osog_device_once.h), compiled for the host:
it runs on every device, once where it succeeds, also from several threads."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_2606_21381_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "osog_device_once.h"
enum Error { kOk = 0, kBad = 3 };
int main() {
    osog::DeviceOnce once;
    int runs[70] = {0}, wrong = 0;
    auto call = [&](int dev, Error e) { return once(dev, [&] { ++runs[dev]; return e; }); };
    wrong += call(0, kOk) != kOk || call(0, kBad) != kOk || runs[0] != 1;   // once
    wrong += call(1, kBad) != kBad || runs[1] != 1;                        // another device
    wrong += call(1, kOk) != kOk || call(1, kBad) != kOk || runs[1] != 2;  // a failure is tried again
    wrong += call(63, kOk) != kOk || call(63, kBad) != kOk || runs[63] != 1;
    wrong += call(69, kOk) != kOk || call(69, kBad) != kBad || runs[69] != 2;  // past the mask: every time
    std::atomic<int> ran{0}, bad{0};
    osog::DeviceOnce shared;
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] {
            for (int i = 0; i < 1000; ++i)
                bad += shared(i % 4, [&] { ++ran; return kOk; }) != kOk;
        });
    for (auto &t : threads) t.join();
    wrong += bad != 0 || ran < 4 || ran > 32;
    std::printf("%d\n", wrong);
    return 0;
}
"""


def test_runs_once_on_each_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "o.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(tmp_path / "o.cpp"), "-o",
                    str(tmp_path / "o")], check=True)
    assert subprocess.run([str(tmp_path / "o")], check=True, capture_output=True,
                          text=True).stdout.strip() == "0"


def test_no_opt_in_is_remembered_for_the_process():
    # cudaFuncSetAttribute acts on the current device: its result is not kept in a
    # function-local static
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+(const\s+)?cudaError_t\s+\w+\s*=", text), name
