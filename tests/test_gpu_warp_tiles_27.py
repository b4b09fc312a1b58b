"""The 27-point step over x tiles one warp wide (variant 5) at the sides where it
can go wrong: rows of one partly filled tile (FP32, 68 to 128) and of several, cut
inside a 64-byte line, tiles of uneven height, runs of one plane (each with its own
prologue and last cubes) and of every length.

One step against the oracle within the stencil's one-step tolerances, then the sums
of the new fields (by cubes) against the oracle's bond sums of the same fields."""
import pytest

from gpu_helpers import compare_states
from oracle.oracle import Oracle
from paper_0911_5692_gb300 import Lattice
from test_gpu_stencil27 import TOL, _check_scalars, _own_sums_check, _params, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(0, 0, 0), (14, 1, 2), (16, 3, 1)])
@pytest.mark.parametrize("prec,n", [(32, 68), (32, 100), (32, 124), (32, 128), (32, 132), (32, 140), (32, 148),
                                    (64, 68), (64, 92), (64, 132)])
def test_ragged_sides(prec, n, shape):
    model = "m2phi2" if n % 8 else "lphi4"
    p = _params(model, n, prec)
    st = _state(model, n, prec, seed=n + shape[0])
    g = Lattice(p)
    if shape[0]:
        g.set_kernel(5, *shape)
    info = g.kernel_info()
    assert info["variant"] == 5 and shape[0] in (0, info["ty"])
    g.set_state(*st, t=0.0, a=1.05, ad=0.5)
    o = Oracle(p)
    o.set_state(*st, t=0.0, a=1.05, ad=0.5)
    g.evolve(1)
    o.step(1)
    compare_states(g, o, TOL[prec], f"N={n} fp{prec} {shape}")
    _check_scalars(g, o, prec, 1)
    o.close()
    _own_sums_check(g, p, prec)
