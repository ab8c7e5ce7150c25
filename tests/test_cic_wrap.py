"""The particle deposit's wrap of positions outside the box, compiled for the host: over
the whole range of FP32 coordinates, not finite ones among them, the cell is in the grid and
the fraction in [0, 1], and up to 2^45 cells it is the position's own (exact remainder,
to the 2^-24 of the fraction and the FP64 rounding of the position in cells)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <cmath>
#include "bsp_cic.h"
int main() {
    const int sizes[] = {8, 10, 54, 150, 256, 512, 1620};
    const double boxes[] = {1.0, 7.3, 1000.0, 2048.0, 1e-3, 3e7};
    unsigned s = 1;
    for (int n : sizes)
        for (double box : boxes)
            for (uint32_t top = 0; top < 1u << 13; ++top)
                for (int k = 0; k < 4; ++k) {
                    s = s * 1664525u + 1013904223u;
                    const uint32_t low = k == 0 ? 0u : k == 1 ? (1u << 19) - 1 : (s >> 8) & ((1u << 19) - 1), bits = top << 19 | low;
                    float p;
                    std::memcpy(&p, &bits, 4);
                    for (int g = 0; g < 2; ++g) {
                        const double u = (double)p * ((double)n / box) - 0.5 * g;
                        int cell;
                        float frac;
                        bsp::cic_wrap(u, n, cell, frac);
                        bool ok = cell >= 0 && cell < n && frac >= 0.f && frac <= 1.f;
                        if (ok && std::fabs(u) < 0x1p45) {
                            double r = std::remainder(u - 0.0, (double)n);   // exact
                            double d = std::remainder((double)cell + (double)frac - r, (double)n);
                            ok = std::fabs(d) <= 0x1p-24 + n * 0x1p-52;
                        }
                        if (!ok) {
                            std::printf("n %d box %g p %.9g grid %d: cell %d fraction %.9g\n", n, box, p, g, cell, frac);
                            return 1;
                        }
                    }
                }
    return 0;
}
"""


def test_wrap_stays_in_the_grid(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "wrap.cpp", tmp_path / "wrap"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1708_05303_gb300", "csrc"), "-o", str(exe), str(src)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
