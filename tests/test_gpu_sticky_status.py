"""A non-finite status stays: every later wait reports it again, and no step, one by one or
as a captured graph, advances the lattice any more."""
import ctypes as C

import numpy as np
import pytest

from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, m2phi2, random_state

pytestmark = pytest.mark.gpu

LAT_ENONFINITE = 5


@pytest.mark.parametrize("prec,n", [(64, 16), (32, 16), (32, 100)])
def test_a_failed_lattice_stays_where_it_is(prec, n):
    # 1 - dt q gamma < 0: the sums pass before the first step finds no real root
    p = lphi4(n, precision=prec)
    g = Lattice(p)
    g.set_state(*random_state(n, 3, precision=prec), t=0.0, a=1.2, ad=-0.7 * 1.2 / p["dt"], step=0)
    before = None
    for steps in (1, 3, 40):
        assert g._L.lat_evolve(g._h, steps) == 0          # queued; the status is the device's
        assert g._L.lat_sync(g._h) == LAT_ENONFINITE
        assert g._L.lat_sync(g._h) == LAT_ENONFINITE
        s = np.empty(8)
        assert g._L.lat_get_scalars(g._h, s.ctypes.data_as(C.POINTER(C.c_double))) == LAT_ENONFINITE
        x = np.empty(n ** 3, dtype=g.np_dtype)
        assert g._L.lat_get_state(g._h, 0, 0, x.ctypes.data_as(C.c_void_p), 0) == LAT_ENONFINITE
        assert s[3] == 0 and s[0] == 0.0
        assert before is None or before == (s.tobytes(), x.tobytes())
        before = (s.tobytes(), x.tobytes())


@pytest.mark.parametrize("expansion", [0, 1])
def test_a_lattice_that_fails_on_its_way_stops_there(expansion):
    p = m2phi2(16, precision=32, expansion=expansion)
    st = random_state(16, 4, precision=32)
    st[0][3, 2, 1] = 1e30                                 # its square is past FP32
    g = Lattice(p)
    g.set_state(*st, t=0.0, a=1.0, ad=0.3 if expansion else 0.0, step=0)
    steps = []
    for _ in range(2):
        g.evolve(5)
        assert g._L.lat_sync(g._h) == LAT_ENONFINITE
        s = np.empty(8)
        assert g._L.lat_get_scalars(g._h, s.ctypes.data_as(C.POINTER(C.c_double))) == LAT_ENONFINITE
        steps.append(s[3])
    assert steps[0] == steps[1] < 5
