"""The averages of an FP32 lattice that do not contain a' (its fields are FP32, its
averages are FP64 sums of them): t, a, the potential and phi's mean to 1e-11 of the
oracle, whatever the side and the model. FP32 sums would leave 1e-7."""
import pytest

from gpu_helpers import paired
from paper_0911_5692_gb300.workloads import lphi4, m2phi2, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stencil", [7, 27])
@pytest.mark.parametrize("model", [lphi4, m2phi2])
@pytest.mark.parametrize("n", [4, 8, 12, 20, 36, 64])
def test_averages_without_the_rate_are_fp64_sums(n, model, stencil):
    p = dict(model(n, precision=32), stencil=stencil)
    st = random_state(n, 31 + n, precision=32, f_mean=(1.0, 0.0), f_amp=(1e-2, 1e-2), pi_mean=(0.4, 0.0),
                      pi_amp=(1e-2, 1e-2))
    g, o = paired(p, st, (0.5, 1.05, 0.6, 0))
    eg, eo = g.energies(), o.energies()
    for k in ("t", "a", "pot", "mean0"):
        assert abs(eg[k] - eo[k]) <= 1e-11 * abs(eo[k]), k
