"""The threads of SS-FULL's host decomposition use next to no processor time while
they wait: beside a serial part of 0.4 s three waiting threads take less than a
quarter of it together (one thread that polls takes all of it), and they are there
for the next step."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1605_07951_gb300", "csrc")

HARNESS = r"""
#include "ssfull_host.cpp"
#include <chrono>
#include <cstdio>
#include <ctime>
int main() {
    rsrr::Workers pool(4);
    std::vector<int> hit(1001, 0);
    auto step = [&]() {
        pool.run(1001, [&](int b, int e) {
            for (int i = b; i < e; ++i) ++hit[i];
        });
    };
    for (int i = 0; i < 3; ++i) step();
    timespec a, b;
    clock_gettime(CLOCK_PROCESS_CPUTIME_ID, &a);
    std::this_thread::sleep_for(std::chrono::milliseconds(400));
    clock_gettime(CLOCK_PROCESS_CPUTIME_ID, &b);
    for (int i = 0; i < 1000; ++i) step();
    std::this_thread::sleep_for(std::chrono::milliseconds(20));
    step();
    int wrong = 0;
    for (int h : hit) wrong += h != 1004;
    printf("%d %.6f\n", wrong, (b.tv_sec - a.tv_sec) + 1e-9 * (b.tv_nsec - a.tv_nsec));
    return 0;
}
"""


def test_waiting_threads_are_idle(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "harness.cpp").write_text(HARNESS)
    exe = str(tmp_path / "idle")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fcx-fortran-rules", "-I", SRC, str(tmp_path / "harness.cpp"), "-o", exe,
                    "-pthread"], check=True, capture_output=True, text=True)
    wrong, cpu = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(wrong) == 0
    assert float(cpu) < 0.1
