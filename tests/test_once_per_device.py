"""What the library does once per device ordinal is asked for by several host threads at once: the helper behind it, built
with ThreadSanitizer from the library's own header."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_34318_b200", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "once_per_device.h"
static hydra::OncePerDevice once;
static std::atomic<int> runs[hydra::kMaxDevices];
int main()
{
    int bad = 0;
    if (once(5, [] { return 3; }) != 3 || once(5, [] { return 3; }) != 3) ++bad;          // a failure is not remembered
    if (once(5, [] { return 0; }) != 0 || once(5, [] { return 3; }) != 0) ++bad;          // success is
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([] {
            for (int i = 0; i < 2000; ++i) once(i % 4, [i] { ++runs[i % 4]; return 0; });
        });
    for (auto& t : threads) t.join();
    for (int d = 0; d < 4; ++d) {
        const int before = runs[d];
        if (before < 1 || before > 8) ++bad;
        once(d, [d] { ++runs[d]; return 0; });
        if (runs[d] != before) ++bad;
    }
    std::printf("done %d\n", bad);
    return bad;
}
"""


def test_once_per_device_from_many_threads(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    build = ["g++", "-std=c++17", "-O1", "-pthread", "-fsanitize=thread", "-I", CSRC, str(src), "-o", str(exe)]
    try:
        built = subprocess.run(build, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no g++")
    if "tsan" in built.stderr and built.returncode:
        pytest.skip("no ThreadSanitizer runtime")
    assert built.returncode == 0, built.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    if "FATAL: ThreadSanitizer" in run.stderr:
        pytest.skip("ThreadSanitizer does not start here: " + run.stderr.strip().splitlines()[0])
    assert run.returncode == 0 and "done 0" in run.stdout, run.stdout + run.stderr
    assert "data race" not in run.stderr, run.stderr
