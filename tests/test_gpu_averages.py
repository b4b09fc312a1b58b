"""The averages and spectra at the sides and bin counts where their kernels' edges
lie (sides of one vector and one pair of rows, z runs of one plane, spectra cut
below and far above the grid's corner, repeated calls on one handle), against the
oracle. Tolerances as in the parity tests of 32^3: FP64 1e-11 (differences of nearby
numbers, the gradient parts and the residual curvature, 1e-10); FP32 lattices hold
the same rounded fields on both sides and sum them in FP64: the same."""
import numpy as np
import pytest

from gpu_helpers import paired
from oracle.oracle import Oracle
from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, m2phi2, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("model", ["lphi4", "m2phi2"])
@pytest.mark.parametrize("n", [4, 8, 12, 20, 36, 64])
def test_energies_at_odd_sides(n, model, prec):
    p = (lphi4 if model == "lphi4" else m2phi2)(n, precision=prec)
    st = random_state(n, 31 + n, precision=prec, f_mean=(1.0, 0.0), f_amp=(1e-2, 1e-2), pi_mean=(0.4, 0.0),
                      pi_amp=(1e-2, 1e-2))
    g, o = paired(dict(p), st, (0.5, 1.05, 0.6, 0))
    eg, eo = g.energies(), o.energies()
    # an FP32 lattice's a' at the field time follows its FP32 sums (2e-6 of a'' at
    # most), which enters the kinetic terms through r h f
    tol = 1e-11 if prec == 64 else 4e-6
    for k in ("t", "a", "ad", "H", "rho", "p", "kin0", "kin1", "pot", "mean0"):
        assert abs(eg[k] - eo[k]) <= tol * max(abs(eo[k]), 1e-3 * abs(eo["rho"]) if k in ("p", "kin0", "kin1") else 0) + 1e-300, k
    for k in ("grad0", "grad1", "var0", "var1"):
        assert abs(eg[k] - eo[k]) <= 1e-10 * abs(eo[k]), k
    assert abs(eg["mean1"] - eo["mean1"]) <= 1e-12 * np.sqrt(eo["var1"])
    again = g.energies()
    assert again == eg


@pytest.mark.parametrize("n", [4, 12, 20, 32])
@pytest.mark.parametrize("prec", [32, 64])
def test_spectrum_bins_at_the_edges(n, prec):
    p = lphi4(n, precision=prec)
    st = random_state(n, 7 * n, precision=prec, f_mean=(1.0, 0.0), f_amp=(1e-3, 1e-3), pi_mean=(0.5, 0.0),
                      pi_amp=(1e-3, 1e-3))
    g = Lattice(p)
    g.set_state(*st, t=0.0, a=1.0, ad=0.5, step=0)
    o = Oracle(p)
    o.set_state(*st, t=0.0, a=1.0, ad=0.5, step=0)
    for bins in (1, n // 2, n, 4096, n):
        for field in (0, 1):
            kg, pg, cg = g.spectrum(field, bins)
            ko, po, co = o.spectrum(field, bins)
            assert np.array_equal(cg, co)
            assert np.allclose(kg, ko, rtol=1e-12, atol=0)
            # phi's mean of 1 leaves about 1e-16 n^(3/2) of its transform in every mode, against
            # amplitudes of 1e-3 n^(3/2): 1e-13 of each, with room for a shell of few modes
            assert np.allclose(pg, po, rtol=1e-9 if field else 1e-8, atol=0)
    if bins >= n:
        assert cg.sum() == n ** 3
