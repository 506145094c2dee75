"""A part that throws on a worker thread of the host pool (or on a helper thread, when the pool is
busy): every other part still runs and the caller gets the exception."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1401_1757_gb300", "csrc")

SRC = r"""
#include "host_parts.h"
#include <chrono>
#include <cstdio>
#include <new>
#include <thread>
#include <vector>

// `T` parts of which those with bad(k) throw; true if all ran once and the exception arrived
template <class Bad>
static bool job(int T, Bad bad) {
    std::vector<std::atomic<int>> hits(T);
    bool any = false, caught = false;
    for (int k = 0; k < T; ++k) any |= bad(k);
    try {
        rsv::run_parts(T, [&](int k) {
            hits[k]++;
            std::this_thread::sleep_for(std::chrono::microseconds(200));   // so that every thread gets parts
            if (bad(k)) throw std::bad_alloc();
        });
    } catch (const std::bad_alloc&) {
        caught = true;
    }
    for (auto& h : hits)
        if (h.load() != 1) return false;
    return caught == any;
}

int main() {
    for (int rep = 0; rep < 20; ++rep) {
        if (!job(16, [](int) { return true; })) { std::printf("FAIL all\n"); return 1; }
        for (int b = 0; b < 16; b += 5)
            if (!job(16, [&](int k) { return k == b; })) { std::printf("FAIL part %d\n", b); return 1; }
        if (!job(16, [](int) { return false; })) { std::printf("FAIL none\n"); return 1; }
    }
    // the pool busy: helper threads
    bool ok[2] = {true, true};
    std::vector<std::thread> callers;
    for (int c = 0; c < 2; ++c)
        callers.emplace_back([&, c] {
            for (int rep = 0; rep < 30; ++rep) ok[c] &= job(8, [&](int k) { return (k + rep) % 3 == 0; });
        });
    for (auto& t : callers) t.join();
    if (!ok[0] || !ok[1]) { std::printf("FAIL concurrent\n"); return 1; }
    // parts inside a part
    std::atomic<int> inner{0};
    try {
        rsv::run_parts(4, [&](int) { rsv::run_parts(4, [&](int j) { inner++; if (j == 3) throw std::bad_alloc(); }); });
        std::printf("FAIL nested\n");
        return 1;
    } catch (const std::bad_alloc&) {
    }
    if (inner.load() != 16) { std::printf("FAIL nested count %d\n", inner.load()); return 1; }
    std::printf("OK\n");
    return 0;
}
"""


def test_parts_that_throw(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "errors.cpp"
    src.write_text(SRC)
    exe = tmp_path / "errors"
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout + out.stderr
