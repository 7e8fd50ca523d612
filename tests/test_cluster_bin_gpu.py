"""Binning by one thread-block cluster against the cooperative kernel (GPU).

Small scenes are binned by a cluster, larger ones by the cooperative kernel;
a scene in a batch with a large one goes the second way.  Its results are the
same bit for bit, at the edges of the blocks' slot and cell ranges, with
crowded cells, agents outside the box, and a second call in the order that
the first recorded (also when the caller permuted its arrays in between).
"""
import numpy as np
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def _filler():
    return scenes.open_square(21000, 230.0, seed=90)


def _check(s, cell=None):
    import torch
    one = api.DeviceScene(s, "cuda", cell_size=cell, debug=True)
    both = api.DeviceBatch([s, _filler()], "cuda", cell_sizes=[cell, None], debug=True)
    for n_steps in (1, 3):
        one.step(n_steps)
        both.step(n_steps)
        torch.cuda.synchronize()
        assert one.sync_status() == 0 and both.sync_status() == 0
        assert torch.equal(one.pos, both.pos[:s.n]) and torch.equal(one.vel, both.vel[:s.n])
        for k in ("cell", "nbr", "cnt", "flags", "tstar"):
            assert torch.equal(one.dbg[k], both.dbg[k][:s.n]), k
    one.close()
    both.close()


@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 2049, 9000, 16385, 20480])
def test_slot_ranges(n):
    _check(scenes.open_square(n, (n / 0.4) ** 0.5 + 1.0, seed=91))


@pytest.mark.parametrize("n, cell", [(512, None), (513, None), (8192, None), (8193, None),
                                     (2000, 1.1), (2000, 1.05), (8192, 0.55)])
def test_block_sizes(n, cell):
    """One agent and more per thread, few and many cells per block."""
    _check(scenes.open_square(n, (n / 0.4) ** 0.5 + 1.0, seed=95), cell)


@pytest.mark.parametrize("cell", [0.19, 0.08, 400.0])
def test_cell_ranges(cell):
    """69k cells (more blocks than the agents need), 391k cells, one cell."""
    _check(scenes.open_square(1500, 50.0, seed=92), cell)


def test_crowded_cells_and_agents_outside_the_box():
    s = scenes.open_square(3000, 60.0, seed=93)
    s.pos[:1200] *= 0.02           # a thousand agents in one cell
    s.pos[2500:] -= 100.0          # outside: clamped to the edge cells
    _check(s)


def test_recorded_order_and_permuted_arrays():
    import torch
    s = scenes.open_square(5000, 110.0, seed=94)
    ds = api.DeviceScene(s, "cuda")
    ds.step(2)
    p = torch.as_tensor(np.random.default_rng(1).permutation(s.n), device="cuda")
    ref = s.copy()
    ref.pos, ref.vel = ds.pos[p].cpu().numpy(), ds.vel[p].cpu().numpy()
    ref.goal = s.goal[p.cpu().numpy()]
    for t in (ds.pos, ds.vel, ds.goal):
        t.copy_(t[p].clone())
    fresh = api.DeviceScene(ref, "cuda")
    ds.step(1)
    fresh.step(1)
    torch.cuda.synchronize()
    assert ds.sync_status() == 0
    assert torch.equal(ds.pos, fresh.pos) and torch.equal(ds.vel, fresh.vel)
    ds.close()
    fresh.close()


def test_nonfinite_input_is_reported():
    s = scenes.open_square(2000, 70.0, seed=95)
    s.vel[1999, 1] = np.nan
    ds = api.DeviceScene(s, "cuda")
    ds.step(1)
    assert ds.sync_status() == 4
    ds.close()
