"""The binning kernel's grid barrier does not give up early (needs a GPU).

The wait that orca.h states (half a second at least) must pass before a step is
given up, and it must end by itself.
"""
import time

import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def test_wait_is_as_long_as_stated():
    import torch
    ds = api.DeviceScene(scenes.open_square(20000, 200.0, seed=11), flags=api.BARRIER_TIMEOUT_TEST)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ds.step(1)
    torch.cuda.synchronize()
    elapsed = time.perf_counter() - t0
    assert ds.sync_status() == 3
    assert 0.5 <= elapsed <= 3.0
    ds.close()
