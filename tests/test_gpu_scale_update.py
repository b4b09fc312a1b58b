"""The scalar update at the end of a step (eq. scale) against the oracle over the
forms it takes: the implicit a' equation far from and near its double root
(1 - dt q gamma below 0.25 and above 4, where the Newton form gives way to the
square root), a' below the FP32 range, powers of a that are not integers, the
homogeneous mode beside it, and blocks of one warp (N = 4) up to many blocks.

Tolerances, FP64: the fields as every one-step parity test (1e-12 normwise); a to
1e-14 and a' to 1e-13 of the larger of |a'| and the fields' scale 1, some hundred
roundings of 1.1e-16 amplified by 1/sqrt(disc) <= 4.
"""
import numpy as np
import pytest

from gpu_helpers import compare_states, paired
from paper_0911_5692_gb300 import Lattice, LatticeError
from paper_0911_5692_gb300.workloads import lphi4, m2phi2, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 16, 36])
@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("form", ["plain", "near root", "near", "far", "tiny", "powers", "m2phi2"])
def test_scalar_update_forms(form, split, n):
    p = m2phi2(n, precision=64, split=split) if form == "m2phi2" else lphi4(n, precision=64, split=split)
    a, unit = 1.2, 1.2 / p["dt"]      # disc = 1 + gamma / unit for lambda phi^4 (q = -1/a), gamma = 2 a' nearly
    ad = {"plain": 0.4, "near root": -0.45 * unit, "near": -0.3 * unit, "far": 2.5 * unit}.get(form, 0.4)
    if form == "tiny":
        p["eight_pi_G"], ad = 1e-40, 0.0
    if form == "powers":
        p.update(A=2.0, B=2e-7, r=1.1, s=-0.8)
    st = random_state(n, 5 + n, precision=64, f_mean=(1.0, 0.0), f_amp=(1e-3, 1e-3), pi_mean=(0.5, 0.0),
                      pi_amp=(1e-3, 1e-3))
    g, o = paired(p, st, (0.0, a, ad, 0))
    # a' at the field time, as the update before the first step solves it
    assert g.energies()["ad"] == pytest.approx(o.energies()["ad"], rel=1e-13, abs=1e-60)
    if form.startswith("near"):       # a collapse: the root is there for this step only
        return
    g.evolve(2)
    o.step(2)
    compare_states(g, o, 1e-12, f"{form} N={n}")
    gs, os_ = g.scalars(), o.scalars()
    assert gs["step"] == os_["step"] == 2
    assert abs(gs["a"] - os_["a"]) <= 1e-14 * max(abs(os_["a"]), abs(os_["ad"]) * p["dt"])
    assert abs(gs["ad"] - os_["ad"]) <= 1e-13 * max(abs(os_["ad"]), 1.0)
    if form == "tiny":                # far below FP32's smallest number, and still right to FP64
        assert 0.0 < os_["ad"] < 1e-38
        assert gs["ad"] == pytest.approx(os_["ad"], rel=1e-12)


def test_scalar_update_reports_no_root():
    """1 - dt q gamma < 0: no real root, a sticky LAT_ENONFINITE as before."""
    p = lphi4(16, precision=64)
    st = random_state(16, 3, precision=64)
    g = Lattice(p)
    g.set_state(*st, t=0.0, a=1.2, ad=-0.7 * 1.2 / p["dt"], step=0)
    with pytest.raises(LatticeError) as e:
        g.evolve(1)
        g.sync()
    assert e.value.status == 5
    assert np.isfinite(g._L.lat_sync(g._h))
