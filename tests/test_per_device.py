"""Kernel attributes are set once for every device of a process, by whichever thread comes first, and again after
a failure (the host logic, with pretended devices)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20686_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    static odgs::PerDevice p;
    int calls = 0;
    auto make = [&](int v) { return [&calls, v] { ++calls; return v; }; };
    CHECK(p.get(0, make(3)) == 3 && p.get(0, make(9)) == 3 && calls == 1);
    CHECK(p.get(1, make(5)) == 5 && calls == 2 && p.get(0, make(9)) == 3 && p.get(1, make(9)) == 5 && calls == 2);
    CHECK(p.get(2, make(0)) == 0 && p.get(2, make(-1)) == -1 && calls == 4);  // failures are tried again
    CHECK(p.get(2, make(7)) == 7 && p.get(2, make(0)) == 7 && calls == 5);
    CHECK(p.get(63, make(2)) == 2 && p.get(64, make(4)) == 4 && p.get(64, make(6)) == 6 && p.get(-1, make(8)) == 8);
    static odgs::PerDevice q;
    std::vector<std::thread> ts;
    std::vector<int> got(16);
    for (int t = 0; t < 16; ++t) ts.emplace_back([&, t] { got[t] = q.get(t % 4, [&] { return 10 + t % 4; }); });
    for (auto& t : ts) t.join();
    for (int t = 0; t < 16; ++t) CHECK(got[t] == 10 + t % 4 && q.get(t % 4, [] { return 1; }) == 10 + t % 4);
    return 0;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_attributes_are_set_through_it():
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        assert "cudaFuncSetAttribute" not in text or "static PerDevice" in text, name
