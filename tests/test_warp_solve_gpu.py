"""The warp-per-agent solve kernel against the per-thread one (needs a GPU).

Small scenes are solved with one warp per agent, larger ones (and the
counting variant at any size) with one thread per agent.  A step's results do
not depend on which ran: every output is compared bit for bit, at the ends of
the neighbour range, with the vehicles' extra half-planes, with exact ties,
and with an agent count on both sides of the dispatch.
"""
import numpy as np
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def _both(s, n_steps=2):
    import torch
    got = []
    for counted in (False, True):
        ds = api.DeviceScene(s, "cuda", debug=True)
        if counted:
            counters = torch.zeros(13, dtype=torch.int64, device="cuda")
            api.orca_scene_set_counters(ds.handle, counters)
        ds.step(n_steps)
        torch.cuda.synchronize()
        assert ds.sync_status() == 0
        got.append({"pos": ds.pos.clone(), "vel": ds.vel.clone(),
                    **{k: v.clone() for k, v in ds.dbg.items()}})
        ds.close()
    for k in got[0]:
        assert torch.equal(got[0][k], got[1][k]), k


def _moving(s, seed):
    rng = np.random.default_rng(seed)
    s.vel = (0.6 * s.max_speed[:, None] * rng.standard_normal((s.n, 2))).astype(np.float32)
    return s


@pytest.mark.parametrize("k", [0, 1, 10, 16, 17, 31, 32])
@pytest.mark.parametrize("n,side", [(1, 5.0), (33, 6.0), (1500, 60.0), (1500, 14.0)])
def test_equals_the_per_thread_kernel(n, side, k):
    s = _moving(scenes.open_square(n, side, seed=70 + k), k)
    s.params.max_neighbors = k
    _both(s)


@pytest.mark.parametrize("k", [10, 13, 14, 29, 30])
def test_vehicle_limits(k):
    s = _moving(scenes.shared_space(n_ped=1500, n_veh=200, side=90.0, seed=71), 5)
    s.params.max_neighbors = k
    s.params.vehicle_turn_rate, s.params.vehicle_accel = 0.8, 2.0
    _both(s)


@pytest.mark.parametrize("tall", [False, True])
@pytest.mark.parametrize("n,k", [(2, 10), (17, 10), (40, 10), (1023, 32), (1024, 10), (1025, 10)])
def test_scenes_without_cells(n, k, tall):
    """The smallest scenes are sorted along the longer side of their box and
    searched without cells, here also with agents outside the box, some at the
    same coordinate, and most beyond the neighbour distance."""
    s = _moving(scenes.open_square(n, 60.0, seed=74 + k), 8)
    s.params.max_neighbors = k
    a, b = (0, 1) if tall else (1, 0)
    s.pos[:, a] *= np.float32(0.2)
    s.pos[: n // 3, b] = s.pos[0, b]
    s.pos[n // 2:, b] *= np.float32(9.0)
    s.params.extent = (12.0, 60.0) if tall else (60.0, 12.0)
    _both(s, 3)


def test_exact_ties():
    """A lattice at rest: equal distances everywhere, equal penetrations."""
    s = scenes.open_square(2500, 40.0, seed=72)
    g = np.stack(np.meshgrid(np.arange(50), np.arange(50)), -1).reshape(-1, 2)
    s.pos = np.ascontiguousarray(0.75 * g, dtype=np.float32)
    _both(s)
    _both(s.subset(np.arange(900)))


@pytest.mark.parametrize("n,k", [(18432, 10), (18433, 10), (28673, 16), (30000, 30)])
def test_both_sides_of_the_dispatch(n, k):
    s = _moving(scenes.open_square(n, (n / 0.4) ** 0.5, seed=73), 6)
    s.params.max_neighbors = k
    _both(s, 1)
