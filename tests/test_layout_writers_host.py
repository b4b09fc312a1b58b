"""The new-field plane that the warps of a block share in the 7-point warp-tile kernel
(lat_xw.cuh): every vector of it has exactly one writer, and the row after a pair's
second is among those written, for each compiled tile (rows whole, several pairs to
a warp, or cut into x tiles) and every side it serves. The places are the kernel's
own (XW::row_of, holds, off_g, shares), compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0911_5692_gb300")

PROGRAM = r'''
#include <cstdio>
#include <map>
#include "lat_xw.cuh"

// one tile: ty rows, qn vectors
template <typename F>
int tile(int n, int ty, int qn)
{
    std::map<unsigned, int> writers;
    for (int w = 0; w <= F::PWARPS; w++) {
        if (w < F::PWARPS && 2 * w * F::RPW >= ty) continue;   // idle
        for (int l = 0; l < 32; l++) {
            const bool ahead = w == F::PWARPS;
            const int pair = F::pair_of(w, l), lx = l % F::LW;
            if (F::shares(F::holds(ahead, pair, l, lx, qn, ty))) writers[F::off_g(F::row_of(ahead, pair, ty), lx)]++;
        }
    }
    for (auto& e : writers)
        if (e.second != 1 || e.first + F::VW > F::FIELDG) { printf("n=%d ty=%d qn=%d offset %u: %d writers\n", n, ty, qn, e.first, e.second); return 1; }
    for (int r = 0; r <= ty / 2; r++)   // the pairs' first rows and the look-ahead row
        for (int q = 0; q < qn; q++)
            if (!writers.count((unsigned)(r * F::W + q * F::VW))) { printf("n=%d ty=%d: row %d vector %d unwritten\n", n, ty, r, q); return 1; }
    return 0;
}

template <typename F>
int whole_rows(int most)
{
    constexpr int TY = 2 * F::PAIRS;
    for (int n = 4; n <= most; n += 4) {
        const int nyt = (n + TY - 1) / TY;
        for (int yt = 0; yt < nyt; yt++) {
            const int ty = 2 * ((yt + 1) * (n / 2) / nyt) - 2 * (yt * (n / 2) / nyt);
            if (tile<F>(n, ty, n / F::VW)) return 1;
        }
    }
    return 0;
}

template <typename F>
int x_tiles()
{
    for (int ty = 2; ty <= 2 * F::PAIRS; ty += 2)
        for (int qn = 1; qn <= 32; qn++)
            if (tile<F>(0, ty, qn)) return 1;
    return 0;
}

int main()
{
    using namespace lat::xw;
    return whole_rows<XW<float, 16, 2, false, 16>>(64) || whole_rows<XW<float, 16, 2, false, 32>>(128) ||
           whole_rows<XW<float, 8, 2, false, 32>>(128) || whole_rows<XW<float, 14, 2, false, 32>>(128) ||
           whole_rows<XW<float, 28, 2, false, 16>>(64) || whole_rows<XW<float, 56, 2, false, 8>>(32) ||
           x_tiles<XW<float, 16, 2, false>>() || x_tiles<XW<double, 4, 1, false>>();
}
'''


def test_every_shared_vector_has_one_writer(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "writers.cu", tmp_path / "writers"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "csrc"), "-I",
                    os.path.join(os.path.dirname(ROOT), "include"), "-o", str(exe), str(src)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
