"""A derivative whose forward pass fails (non-finite sums) leaves the lattice as
lat_evolve does: at the step that failed, with that step's fields, momenta and
scalars and the sticky status; and it writes no value of the observable. The
failing step lies at the start, inside and at the end of the last checkpoint
segment, and before it, at odd and even distances from the last step. Compared byte
for byte: both run the same step kernel from the same state."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, random_state

pytestmark = pytest.mark.gpu

LAT_ENONFINITE = 5


def _lattice(n, prec, odd):
    # far outside the stable range (dt^2 3 f^2 > 4): f grows like dt^2 f^3 per step
    # until the sums overflow
    p = lphi4(n, precision=prec, expansion=0)
    big = 2.0 / p["dt"]
    st = random_state(n, 7, prec, f_mean=(big, 0.0), f_amp=(0.1 * big, 1e-3), pi_mean=(0.0, 0.0), pi_amp=(1e-3, 1e-3))
    g = Lattice(p)
    g.set_state(*st, t=0.0, a=1.0, ad=0.0, step=odd)
    return g


def _snapshot(g):
    out = []
    for what in (0, 1):
        for field in (0, 1):
            x = np.empty(g.n ** 3, dtype=g.np_dtype)
            assert g._L.lat_get_state(g._h, field, what, x.ctypes.data_as(C.c_void_p), 0) == LAT_ENONFINITE
            out.append(x.tobytes())
    s = np.empty(8)
    assert g._L.lat_get_scalars(g._h, s.ctypes.data_as(C.POINTER(C.c_double))) == LAT_ENONFINITE
    return out, s


@pytest.mark.parametrize("call", ["chi2", "fraction", "vjp"])
@pytest.mark.parametrize("n,prec,odd", [(16, 64, 0), (16, 32, 1), (64, 32, 0)])
def test_failed_forward_pass_leaves_the_state_reached(n, prec, odd, call):
    ref = _lattice(n, prec, odd)
    reached = 0
    while ref._L.lat_sync(ref._h) == 0:
        ref.evolve(1)
        reached += 1
        assert reached < 30
    assert reached >= 3
    fields, scalars = _snapshot(ref)
    assert scalars[3] == odd + reached
    for beyond in (0, 1, 2, 3):
        steps = reached + beyond
        # one segment; the failing step last and first of the last segment; and before it
        for every in {steps, (steps + 1) // 2, max(1, reached - 1), reached, 1}:
            g = _lattice(n, prec, odd)
            bars = [torch.zeros(2 * n ** 3, dtype=g.dtype, device="cuda") for _ in range(2)]
            torch.cuda.synchronize()
            ptr = [C.c_void_p(b.data_ptr()) for b in bars]
            J, dg2 = C.c_double(-7.0), C.c_double(-7.0)
            if call == "vjp":
                st = g._L.lat_vjp(g._h, steps, every, *ptr, (C.c_double * 4)())
            else:
                st = g._L.lat_adjoint(g._h, steps, int(call == "fraction"), every, C.byref(J), C.byref(dg2), *ptr)
            assert st == LAT_ENONFINITE
            assert J.value == -7.0 and dg2.value == -7.0
            got, s = _snapshot(g)
            assert s.tobytes() == scalars.tobytes(), (steps, every)
            assert got == fields, (steps, every, [a == b for a, b in zip(got, fields)])
            g.close()
