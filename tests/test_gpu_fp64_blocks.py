"""The automatic FP64 shape of 7-point lattices below 256^3: one block to an SM at most
(several are not spread evenly over the SMs), no block with more plane steps than a
full wave of that tile height has, and one step equal bit for bit in fields and
momenta to that of an explicit shape."""
import numpy as np
import pytest
import torch

from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4, random_state

pytestmark = pytest.mark.gpu


def _busiest(n, nyt, blocks):
    most = 0
    for b in range(blocks):
        u, e = b * nyt * n // blocks, (b + 1) * nyt * n // blocks
        most = max(most, e - u + (e - 1) // n - u // n + 1)
    return most


def test_one_block_to_an_sm_and_no_longer_share():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in list(range(4, 132, 4)) + [160, 200, 252]:
        info = Lattice(lphi4(n, precision=64)).kernel_info()
        assert info["variant"] == 2 and info["depth"] == 1
        nyt, blocks = n // info["ty"], info["blocks"]
        assert 1 <= blocks <= sms, (n, info)
        assert _busiest(n, nyt, blocks) <= _busiest(n, nyt, min(sms, nyt * n)), (n, info)


@pytest.mark.parametrize("n", [4, 12, 20, 36, 40, 52, 60, 68, 72, 76, 80, 100, 108])
def test_a_step_equals_that_of_an_explicit_shape(n):
    st = random_state(n, 9, 64, f_mean=(1.0, 0.0), f_amp=(1e-3, 1e-3), pi_mean=(0.5, 0.0), pi_amp=(1e-3, 1e-3))
    out = []
    for shape in ((0, 0, 0, 0), (2, 4, 0, 1), (2, 2, 3, 2)):
        g = Lattice(lphi4(n, precision=64))
        g.set_kernel(*shape)
        g.set_state(*st, t=0.0, a=1.1, ad=0.4, step=0)
        g.evolve(1)
        out.append((g.get_state(), g.scalars()))
    for state, s in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(state, out[0][0]))
        assert s["ad"] == pytest.approx(out[0][1]["ad"], rel=1e-13)
