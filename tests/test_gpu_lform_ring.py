"""The L = 1/H form's sums pass over the plane ring (FP32) at the sides where it can
go wrong: fewer rows than a tile, rows of one partly filled tile and of several,
cut inside a 64-byte line, tiles of uneven height, runs of one or two planes, both
Laplacians, phi whole and split. Two steps against the oracle within the tolerances of the form's parity
tests, per step."""
import pytest

from gpu_helpers import compare_states, paired
from test_gpu_lform import TOL, _check_scalars, _params, _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("n,stencil", [(n, 7) for n in (4, 12, 20, 36, 56, 60, 68, 100, 128, 132, 148, 260)]
                         + [(n, 27) for n in (4, 12, 20, 68, 100, 128, 132, 148)])
def test_two_steps(n, stencil, split):
    model = "m2phi2" if n % 8 else "lphi4"
    p = dict(_params(model, n, 32, stencil), split=split)
    st = _state(model, n, 32, seed=n + split)
    g, o = paired(p, st, (0.0, 1.1, 0.45, 0))
    for k in (1, 2):
        g.evolve(1)
        o.step(1)
        compare_states(g, o, k * TOL[32], f"L form N={n} split={split} step {k}")
        _check_scalars(g, o, 32, k)
