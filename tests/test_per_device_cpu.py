"""Shared-memory opt-ins are made on every device that a process uses, not once a
process: the class that remembers them, driven on the host, and the sources' use of it."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_12629_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
int main() {
    cube2::PerDevice once;
    int calls[80] = {};
    auto set = [&](int dev, int result) { return once.once(dev, [&] { ++calls[dev]; return result; }); };
    int bad = 0;
    bad += set(0, 0) != 0 || set(0, 0) != 0 || calls[0] != 1;      // once
    bad += set(1, 7) != 7 || set(1, 0) != 0 || set(1, 7) != 0 || calls[1] != 2;   // again after a failure
    bad += set(63, 0) != 0 || set(63, 0) != 0 || calls[63] != 1;
    bad += set(70, 0) != 0 || set(70, 0) != 0 || calls[70] != 2;   // not remembered
    std::atomic<int> made[8] = {};
    std::vector<std::thread> threads;
    cube2::PerDevice shared;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] {
            for (int k = 0; k < 800; ++k) shared.once(k % 8, [&] { ++made[k % 8]; return 0; });
        });
    for (auto &t : threads) t.join();
    for (auto &m : made) bad += m < 1 || m > 8;
    std::printf("%d\n", bad);
}
"""


def test_once_per_device(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    src, exe = str(tmp_path / "once.cpp"), str(tmp_path / "once")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, src, "-o", exe], check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split() == ["0"]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_no_opt_in_is_remembered_for_the_process(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert not re.search(r"static\s+bool", text)
    assert "cudaFuncSetAttribute" not in text    # allow_shared() of common.cuh, inside a PerDevice
    assert text.count("allow_shared(") == 0 or "static PerDevice" in text
