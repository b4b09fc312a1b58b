"""The runs of the 7-point warp-tile step kernel's block groups (TileWalk in
lat_layout.cuh), compiled for the host: every (y tile, z plane) unit is marched by
exactly one group for tile counts below, at and above the group count, runs taken
whole or in parts; and no group has more than the even share allows."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0911_5692_gb300", "csrc")

PROGRAM = r'''
#include <algorithm>
#include <cstdio>
#include <vector>
#include "lat_layout.cuh"

static int check(int T, int G, int zn, int part, double* most)
{
    std::vector<int> cover((size_t)T * zn, 0);
    *most = 0;
    for (int g = 0; g < G; g++) {
        lat::TileWalk w(T, G, g, zn);
        int yt, z0, nz, load = 0, steps = 0;
        while (w.run(yt, z0, nz)) {
            if (part) nz = std::min(nz, part - z0 % part);   // as a z-slab's ranges cut it
            if (yt < 0 || yt >= T || z0 < 0 || nz < 1 || z0 + nz > zn || ++steps > 4 * T * zn) return 1;
            for (int z = z0; z < z0 + nz; z++) cover[(size_t)yt * zn + z]++;
            w.took(nz);
            load += nz;
        }
        *most = std::max(*most, (double)load);
    }
    for (int c : cover)
        if (c != 1) return 1;
    *most /= (double)T * zn / G;
    return 0;
}

int main()
{
    double s;
    for (int T : {1, 2, 5, 7, 9, 16, 19, 24, 36, 64, 128})
        for (int G = 1; G <= 160; G += G < 40 ? 1 : 7)
            for (int zn : {1, 2, 3, 5, 16, 31, 100})
                for (int part : {0, 1, 6})
                    if (check(T, G, zn, part, &s)) { printf("bad T=%d G=%d zn=%d part=%d\n", T, G, zn, part); return 1; }
    // (tiles, groups, planes): 1024^3, 576^3, 384^3, 256^3 and 100^3
    const int cases[5][3] = {{64, 19, 1024}, {36, 30, 576}, {24, 50, 384}, {16, 76, 256}, {7, 152, 100}};
    for (auto& c : cases) {
        if (check(c[0], c[1], c[2], 0, &s)) return 1;
        printf("most %.4f\n", s);
    }
    return 0;
}
'''


def test_walk_covers_every_unit_once(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "walk.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "walk"
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    most = [float(line.split()[1]) for line in out.stdout.splitlines()]
    # the busiest group's planes over the even share: 5 planes where 4.6 are even (100^3) at worst
    assert len(most) == 5 and max(most) <= 1.09, most
