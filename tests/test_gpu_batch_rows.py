"""Ensembles stepped over whole rows (FP32 members of sides up to 128): rows of one,
two and four to a warp with partly filled lanes, tiles of uneven height, members
smaller than a block's share and larger, phi stored split beside whole.

After one step fields and momenta equal those of the same lattices stepped one by
one on the plane-ring kernel bit for bit (the same sums pass sets the
coefficients, every kernel rounds a site alike). After five more the bounds are
those of the one-step parity tests against the oracle, per step: fields 2e-6, a
1e-8, a' 1e-7 (an FP32 lattice's sums, in one order or another, carry about 1e-7,
which moves a' by dt dc with dt up to 0.125 at N = 4).
"""
import numpy as np
import pytest

from paper_0911_5692_gb300 import Ensemble, Lattice
from paper_0911_5692_gb300.workloads import lphi4, m2phi2

pytestmark = pytest.mark.gpu


def _arrays(p, seed):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    a = [torch.randn(p["n"] ** 3, generator=gen, device="cuda", dtype=torch.float32).mul_(1e-3) for _ in range(4)]
    if not p["split"]:
        a[0] += 1.0
        a[2] += 0.4
    torch.cuda.synchronize()
    return a


def _load(g, p, arrays):
    g.set_scalars(t=0.0, a=1.1, ad=0.4, step=0)
    if p["split"]:
        g.set_background(1.0, 0.4)
    g.upload_state(*arrays)
    g.sync()


@pytest.mark.parametrize("sizes,rows", [((4, 20, 28, 32), True), ((36, 52, 64, 32), True), ((68, 100, 128, 96), True),
                                        ((4, 128), True), ((128,), True), ((32, 132), False)])
@pytest.mark.parametrize("copies", [1, 9])
def test_members_equal_single_lattices(sizes, rows, copies):
    import torch
    ps = []
    for i, n in enumerate(sizes * copies):
        ps.append((m2phi2 if i % 3 == 1 else lphi4)(n, precision=32, split=i % 2))
    ens = Ensemble(ps)
    assert (ens.info()["threads"] == 256 and ens.info()["ty"] == [2] * len(ps)) == rows
    states = [_arrays(p, 5 + i) for i, p in enumerate(ps)]
    for i, p in enumerate(ps):
        _load(ens.member(i), p, states[i])
    out = []
    for steps in (1, 5):
        ens.evolve(steps)
        ens.sync()
        for i, p in enumerate(ps):
            t = [torch.empty(p["n"] ** 3, dtype=torch.float32, device="cuda") for _ in range(4)]
            ens.member(i).download_state(*t)
            out.append((t, ens.member(i).scalars()))
    for i, p in enumerate(ps):
        g = Lattice(p)
        g.set_kernel(2)
        _load(g, p, states[i])
        for k, steps in enumerate((1, 5)):
            g.evolve(steps)
            s = g.scalars()
            t, se = out[k * len(ps) + i]
            own = g.buffers[4 * (s["step"] & 1):][:4]
            for x, y in zip(t, own):
                if k == 0:
                    assert torch.equal(x, y)
                else:
                    assert float((x - y).abs().max()) <= 5 * 2e-6 * float(y.abs().max())
            assert se["step"] == s["step"] and se["t"] == s["t"]
            n = se["step"]
            assert abs(se["a"] - s["a"]) <= n * 1e-8 * s["a"] and abs(se["ad"] - s["ad"]) <= n * 1e-7
            assert np.allclose(se["S"], s["S"], rtol=2e-6 if k == 0 else 2e-5)
        g.close()
