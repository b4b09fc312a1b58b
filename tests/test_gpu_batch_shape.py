"""The launch shape an ensemble reports is the one that set_shape takes back: threads,
tile cap and depth given to lat_batch_set_shape select the same kernel, tiles and
blocks, for the default shape, a shape set by hand and the tuned one. A cap of 0
names the whole-row kernel, and is refused where that kernel cannot serve."""
import pytest

from paper_0911_5692_gb300 import Ensemble, LatticeError
from paper_0911_5692_gb300.workloads import lphi4

pytestmark = pytest.mark.gpu

KEYS = ("blocks", "threads", "smem", "ranges", "ty", "tile_cap", "depth")


def _shape(ens):
    info = ens.info()
    return {k: info[k] for k in KEYS}


@pytest.mark.parametrize("prec,sizes", [(32, (32, 48, 64, 96)), (32, (4, 36, 128)), (32, (32, 132)), (64, (32, 48))])
def test_a_reported_shape_can_be_set_again(prec, sizes):
    ens = Ensemble([lphi4(n, precision=prec) for n in sizes])
    default = _shape(ens)
    rows = prec == 32 and max(sizes) <= 128
    assert (default["tile_cap"] == 0) == rows
    shapes = [default]
    ens.set_shape(256, 8, 1)
    shapes.append(_shape(ens))
    assert shapes[1] != default and shapes[1]["tile_cap"] == 8
    ens.init_fields()
    ens.tune(2)
    shapes.append(_shape(ens))
    for want in shapes + shapes[::-1]:
        ens.set_shape(want["threads"], want["tile_cap"], want["depth"])
        assert _shape(ens) == want
    ens.evolve(1)
    ens.sync()
    for args, status in (((256, 0, 1), 1), ((512, 0, 2), 1), ((256, -1, 2), 1)) + (() if rows else (((256, 0, 2), 7),)):
        before = _shape(ens)
        with pytest.raises(LatticeError) as e:
            ens.set_shape(*args)
        assert e.value.status == status and _shape(ens) == before
