"""Every compiled shape of the warp-tile kernel (variant 5) that a lattice can take by
hand is one that its tuner times: the FP64 tiles of 8 and 4 rows among them."""
import pytest

from paper_0911_5692_gb300 import Lattice, LatticeError
from paper_0911_5692_gb300.workloads import lphi4

pytestmark = pytest.mark.gpu

SHAPES = ([(5, ty, d) for ty in (16, 8, 4) for d in (1, 2, 3)] + [(4, ty, d) for ty in (32, 16, 8) for d in (1, 2)] +
          [(2, ty, d) for ty in (16, 8, 4, 2) for d in (1, 2)])


@pytest.mark.parametrize("n,prec", [(24, 64), (56, 64), (68, 32)])
def test_every_shape_that_can_be_set_is_timed(n, prec):
    def launch(g):
        i = g.kernel_info()
        return tuple(i[k] for k in ("variant", "ty", "depth", "blocks", "threads"))

    g = Lattice(lphi4(n, precision=prec))
    launches = {launch(g)}
    for variant, ty, depth in SHAPES:
        try:
            g.set_kernel(variant, ty, 0, depth)
        except LatticeError:
            continue
        launches.add(launch(g))
    assert (prec == 32) or {(5, 8, 1), (5, 4, 1)} <= {x[:3] for x in launches}
    g.set_kernel(0)
    g.init_fields()
    assert g.tune(4)["candidates"] == len(launches)
