"""The tuner times the automatic shape beside the explicit ones, and a tuning that fails
leaves the launch that was in use. In FP64 the automatic block count follows from a
cost rule that no explicit shape reproduces, so neither can be had from the
reported (variant, ty, zr, depth)."""
import pytest

from paper_0911_5692_gb300 import Lattice, LatticeError
from paper_0911_5692_gb300.workloads import lphi4, random_state

pytestmark = pytest.mark.gpu

# every explicit shape the tuner is documented to sweep (variant, ty, depth)
SHAPES = ([(5, 16, d) for d in (1, 2, 3)] + [(5, 8, d) for d in (2, 3)] + [(4, ty, d) for ty in (32, 16, 8) for d in (1, 2)] +
          [(2, ty, d) for ty in (16, 8, 4, 2) for d in (1, 2)])


def _launch(g):
    i = g.kernel_info()
    return tuple(i[k] for k in ("variant", "ty", "depth", "blocks", "threads"))


@pytest.mark.parametrize("n,prec", [(40, 64), (100, 64), (56, 32), (20, 32)])
def test_the_automatic_shape_is_a_candidate(n, prec):
    p = lphi4(n, precision=prec)
    g = Lattice(p)
    automatic = _launch(g)
    launches = {automatic}
    for variant, ty, depth in SHAPES:
        try:
            g.set_kernel(variant, ty, 0, depth)
        except LatticeError:
            continue
        launches.add(_launch(g))
    explicit = len(launches) - 1
    g.set_kernel(0)
    assert _launch(g) == automatic
    g.init_fields()
    r = g.tune(4)
    assert r["candidates"] >= len(launches) >= explicit
    assert _launch(Lattice(p)) == _launch(g)      # a later handle starts with the launch that won


@pytest.mark.parametrize("n", [40, 100, 128])
def test_a_failed_tuning_keeps_the_launch(n):
    p = lphi4(n, precision=64, expansion=0)
    # far outside the stable range: the sums overflow within a few steps
    big = 2.0 / p["dt"]
    st = random_state(n, 3, 64, f_mean=(big, 0.0), f_amp=(0.1 * big, 1e-3), pi_mean=(0.0, 0.0), pi_amp=(1e-3, 1e-3))
    g = Lattice(p)
    g.set_state(*st, t=0.0, a=1.0, ad=0.0, step=0)
    before, fields = g.kernel_info(), g.get_state()
    with pytest.raises(LatticeError) as e:
        g.tune(4)
    assert e.value.status == 5
    assert g.kernel_info() == before
    for x, y in zip(g.get_state(), fields):
        assert (x == y).all()
    assert g.kernel_info() == Lattice(p).kernel_info()
