"""The z runs of the column-marching passes (balanced_zruns in lat_grid.h), compiled for
the host: the count never lets a run fall below the shortest one worth starting, no
other count leaves the busiest thread less to do, and a lattice with fewer columns
than threads is cut down to runs of that length (one plane for the energy sums)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0911_5692_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include "lat_grid.h"

int main()
{
    for (int least : {1, 4})
        for (int n = 4; n <= 1024; n += n < 128 ? 4 : 60)
            for (int v : {2, 4})
                for (double startup : {0.3, 2.0}) {
                    const long long cols = (long long)(n / v) * (n / 2), threads = 152 * 256;
                    auto cost = [&](int c) { return (double)((cols * c + threads - 1) / threads) * ((double)n / c + startup); };
                    const int c = lat::balanced_zruns(cols, n, threads, startup, least);
                    bool ok = c >= 1 && c <= n / least;
                    for (int k = 1; k <= n / least; k++) ok = ok && cost(c) <= cost(k);
                    if (cols * (n / least) <= threads) ok = ok && c == n / least;
                    if (!ok) { printf("n=%d v=%d startup=%g least=%d: %d\n", n, v, startup, least, c); return 1; }
                }
    return 0;
}
'''


def test_runs_are_balanced(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "grid.cu", tmp_path / "grid"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
