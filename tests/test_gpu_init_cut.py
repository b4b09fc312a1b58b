"""Initial fluctuations at the edges of the spectral cut: a cut on, just below and
just above a shell (compared as an integer on the device), between the default and
the grid's corner (the transforms along y and z then take every kx), beyond it, and
so low that one shell is left; both Laplacians, sides with and without a radix of
two, against the oracle. Tolerances as in the default cut's tests: fluctuations of
chi 1e-12 normwise (FP64 transforms of 16^3 to 24^3 values)."""
import math

import numpy as np
import pytest

from gpu_helpers import compare_states, normwise
from oracle.oracle import Oracle
from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, m2phi2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stencil", [7, 27])
@pytest.mark.parametrize("n", [16, 20, 24])
@pytest.mark.parametrize("cut", [1.0, math.sqrt(2.0), math.nextafter(math.sqrt(5.0), 0.0), "quarter", "half", "over half",
                                 "corner", 1e6])
def test_init_parity_at_the_cut(cut, n, stencil):
    kcut = {"quarter": 0.0, "half": n / 2, "over half": n / 2 + 0.5, "corner": math.sqrt(3.0) * n / 2}.get(cut, cut)
    p = dict((lphi4 if n != 20 else m2phi2)(n, precision=64, seed=77 + n), kcut=kcut, stencil=stencil)
    g = Lattice(p)
    g.init_fields()
    o = Oracle(p)
    o.init_fields()
    compare_states(g, o, 1e-13, f"init N={n} kcut={kcut}")
    gs, os_ = g.get_state(), o.get_state()
    for i in (1, 3):
        assert normwise(gs[i], os_[i]) < 1e-12
        assert np.max(np.abs(os_[i])) > 0.0
