"""Removal at goal over the block ranges of its two passes (needs a GPU).

Every agent array is compacted in order, at the edges of a block's tile and
with more agents than one tile for each of the most blocks, with none, some and
all agents at their goal.
"""
import numpy as np
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1023, 1025, 5000, 4096 * 1024 + 3])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_ranges(n, share):
    import torch
    if n > 1000000 and share != 0.3:
        pytest.skip("one share is enough at this size")
    rng = np.random.default_rng(n)
    s = scenes.open_square(n, (n / 0.4) ** 0.5 + 30.0, seed=80)
    s.goal = np.ascontiguousarray(s.goal + np.float32(5000.0))
    arrived = rng.random(n) < share
    s.goal[arrived] = s.pos[arrived]
    s.vel = rng.standard_normal((n, 2)).astype(np.float32)
    ds = api.DeviceScene(s, "cuda", cell_size=8.0)
    kept = ds.remove_arrived()
    want = np.nonzero(~arrived)[0]
    assert np.array_equal(kept, want) and ds.n == len(want)
    for t, a in ((ds.pos, s.pos), (ds.vel, s.vel), (ds.goal, s.goal), (ds.radius, s.radius),
                 (ds.max_speed, s.max_speed), (ds.type, s.type)):
        assert np.array_equal(t[:ds.n].cpu().numpy(), a[want])
    if ds.n:
        ds.step(1)
        torch.cuda.synchronize()
        assert ds.sync_status() == 0
    ds.close()
