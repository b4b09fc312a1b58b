"""Device memory of lat_init_fields while it runs: the noise, two filtered arrays and the
half spectrum (four arrays of N^3 doubles), and one work area for its transforms. On a
side with a large prime factor the transforms along x work in two such arrays
(cuFFT's figure), so six in all; with a work area each it was eight. The free memory
is read every millisecond beside the call."""
import gc
import threading
import time

import pytest
import torch

from paper_0911_5692_gb300 import Lattice
from paper_0911_5692_gb300.workloads import lphi4

pytestmark = pytest.mark.gpu


def test_transforms_share_one_work_area():
    n = 524   # 4 * 131
    g = Lattice(lphi4(n, precision=32))
    small = Lattice(lphi4(32, precision=32))
    small.init_fields()       # what the library sets up once is there
    gc.collect()              # no other test's lattice is freed meanwhile
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = low = torch.cuda.mem_get_info()[0]
    done = threading.Event()
    seen = []

    def watch():
        while not done.is_set():
            seen.append(torch.cuda.mem_get_info()[0])
            time.sleep(1e-3)

    t = threading.Thread(target=watch)
    t.start()
    g.init_fields()
    done.set()
    t.join()
    low = min(seen)
    array = 8 * n ** 3
    assert len(seen) >= 5
    assert 4 * array < before - low < 6.5 * array, (before - low) / array
