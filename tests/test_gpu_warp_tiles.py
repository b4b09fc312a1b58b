"""The step over x tiles one warp wide (variant 5) at the sides where it can go
wrong: rows of one partly filled tile and of several, tiles of fewer rows than the
height (a last pair of rows), rows that split a 32-byte sector between tiles, runs
shorter than the prefetch depth, and more tiles than block groups.

One step from the same state: the coefficients come from the same sums pass, and
every kernel rounds a site's kick and drift alike, so fields and momenta equal the
plane-ring kernel's bit for bit. The sums add the same FP32 (FP64) terms in another
order: 2e-6 (1e-11) relative as in the parity tests."""
import numpy as np
import pytest

from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, m2phi2

pytestmark = pytest.mark.gpu

SHAPES = {32: [(16, 1), (16, 2), (16, 3), (8, 2), (8, 3)], 64: [(16, 1), (16, 2), (8, 1), (4, 1)]}


def _pair(p, other, shape):
    import torch
    out = []
    for variant, ty, depth in ((other, 0, 0), (5, *shape)):
        g = Lattice(p)
        g.set_kernel(variant, ty, 0, depth)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(11)
        arrays = [torch.randn(p["n"] ** 3, generator=gen, device="cuda", dtype=g.dtype).mul_(1e-3) for _ in range(4)]
        if not p["split"]:
            arrays[0] += 1.0
            arrays[2] += 0.4
        torch.cuda.synchronize()
        g.set_scalars(t=0.0, a=1.1, ad=0.4, step=0)
        if p["split"]:
            g.set_background(1.0, 0.4)
        g.upload_state(*arrays)
        g.evolve(1)
        s = g.scalars()
        out.append(([b.clone() for b in g.buffers[4:]], s))
        g.close()
    return out


def _same(p, other, shape):
    import torch
    (a, sa), (b, sb) = _pair(p, other, shape)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    tol = 2e-6 if p["precision"] == 32 else 1e-11
    for x, y in zip(sa["S"], sb["S"]):
        assert abs(x - y) <= tol * abs(x)
    assert sa["a"] == sb["a"] and np.isfinite(sb["ad"])


@pytest.mark.parametrize("shape", range(5))
@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [4, 20, 52, 68, 100, 132, 148, 260])
def test_one_step_equals_the_plane_ring(n, prec, shape):
    if shape >= len(SHAPES[prec]):
        pytest.skip("no such shape")
    model = m2phi2 if n % 8 else lphi4
    _same(model(n, precision=prec, split=int(n % 16 == 4)), 2, SHAPES[prec][shape])


@pytest.mark.parametrize("n,shape", [(516, (8, 3)), (520, (16, 2))])
def test_more_tiles_than_groups(n, shape):
    _same(lphi4(n, precision=32, split=1), 2, shape)
