"""The per-device set-up of kernel attributes (csrc/device_once.h), compiled
for the host: once on every device of a process, again after a failure, and
from several threads."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_40159_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main()
{
    spt::DeviceOnce once, other;
    int calls = 0;
    auto ok = [&] { ++calls; return 0; };
    CHECK(once.run(0, ok) == 0 && calls == 1);
    CHECK(once.run(0, ok) == 0 && calls == 1);
    CHECK(once.run(1, ok) == 0 && calls == 2);  // another device of the process
    CHECK(once.run(63, ok) == 0 && once.run(63, ok) == 0 && calls == 3);
    CHECK(once.run(64, ok) == 0 && once.run(64, ok) == 0 && calls == 5);
    CHECK(once.run(0, ok) == 0 && once.run(1, ok) == 0 && calls == 5);
    CHECK(other.run(0, ok) == 0 && calls == 6);
    int tries = 0;
    auto late = [&] { return ++tries < 3 ? 7 : 0; };
    CHECK(other.run(2, late) == 7 && other.run(2, late) == 7 && other.run(2, late) == 0);
    CHECK(other.run(2, late) == 0 && tries == 3);
    spt::DeviceOnce shared;
    std::vector<std::thread> ts;
    std::vector<int> seen(8, 0);
    for (int t = 0; t < 8; ++t) ts.emplace_back([&, t] { for (int d = 0; d < 32; ++d) shared.run(d, [&] { ++seen[t]; return 0; }); });
    for (auto &t : ts) t.join();
    int sum = 0;
    for (int v : seen) sum += v;
    CHECK(sum >= 32);
    for (int d = 0; d < 32; ++d) CHECK(shared.run(d, [&] { return 1; }) == 0);
    return 0;
}
"""


def test_device_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
