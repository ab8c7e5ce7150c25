"""The shared-memory limits of kernels are attributes per device that setting can lower:
a size asked for on one device must still be set on another, and a smaller size that
comes later, or at the same time in another thread, must not take a larger one back.
The header's bookkeeping is compiled for the host against attributes that only record."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "bsp_smem.h"
static size_t attr[70];
static int calls = 0;
static bsp::SmemLimit limit;
static int ask(int dev, size_t bytes, int err = 0) {
    return limit.raise<int>(dev, bytes, [&](size_t b) { ++calls; if (!err) attr[dev] = b; return err; });
}
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    CHECK(ask(0, 100000) == 0 && attr[0] == 100000 && calls == 1);
    CHECK(ask(0, 60000) == 0 && attr[0] == 100000 && calls == 1);    // smaller: nothing
    CHECK(ask(1, 60000) == 0 && attr[1] == 60000 && calls == 2);     // another device: its own
    CHECK(ask(1, 100000, 7) == 7 && ask(1, 100000) == 0 && attr[1] == 100000);   // a failure is not kept
    CHECK(ask(66, 90000) == 0 && ask(66, 60000) == 0 && attr[66] == 90000);      // past the table: never lowered
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([k] { for (int i = 0; i < 2000; ++i) ask(2, 50000 + 8 * ((i * 7919 + k * 104729) % 20000)); });
    for (auto& x : t) x.join();
    size_t most = 0;
    for (int k = 0; k < 8; ++k) for (int i = 0; i < 2000; ++i) { size_t b = 50000 + 8 * ((i * 7919 + k * 104729) % 20000); if (b > most) most = b; }
    CHECK(attr[2] == most);
    return 0;
}
"""


def test_limits_per_device_and_only_raised(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_1708_05303_gb300", "csrc"), "-o", str(exe),
                    str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_limit_goes_through_it():
    csrc = os.path.join(ROOT, "paper_1708_05303_gb300", "csrc")
    for name in os.listdir(csrc):
        text = open(os.path.join(csrc, name)).read()
        assert text.count("cudaFuncSetAttribute") == (1 if name == "bsp_internal.h" else 0), name
