"""csrc/pp_per_device.h, compiled for the host: one result for each device, worked out
again after a failure, and not mixed up between threads."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_10252_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include <thread>
#include <vector>
#include "pp_per_device.h"
#define CHECK(x) if (!(x)) { printf("line %d: %s\\n", __LINE__, #x); return 1; }
int main() {
    pp::PerDevice a, b;
    int calls = 0;
    for (int round = 0; round < 3; ++round)
        for (int d = 0; d < 4; ++d) CHECK(a.get(d, [&] { ++calls; return 10 * d; }) == 10 * d);
    CHECK(calls == 4);                                            // once on each device
    CHECK(b.get(2, [] { return 7; }) == 7);                       // of its own
    CHECK(a.get(5, [] { return -3; }) == -3);                     // a failure is not kept
    CHECK(a.get(5, [] { return 1; }) == 1);
    CHECK(a.get(5, [] { return 2; }) == 1);
    for (int d : {-1, 64, 1000}) {                                // not kept, but answered
        CHECK(a.get(d, [] { return 1; }) == 1);
        CHECK(a.get(d, [] { return 2; }) == 2);
    }
    pp::PerDevice c;
    std::vector<std::thread> t;
    std::atomic<int> wrong(0);
    for (int i = 0; i < 8; ++i)
        t.emplace_back([&, i] {
            for (int k = 0; k < 1000; ++k)
                if (c.get((i + k) % 64, [&] { return (i + k) % 64; }) != (i + k) % 64) ++wrong;
        });
    for (auto& x : t) x.join();
    CHECK(wrong == 0);
    return 0;
}
"""


def test_results_are_kept_by_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_launch_attributes_are_not_kept_by_process():
    """No function-local static holds what CUDA said about the first device."""
    import re
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static (const )?(cudaError_t|bool) \w+ = (\[|cudaFunc|cudaOcc)", text), name
        assert "call_once" not in text, name
