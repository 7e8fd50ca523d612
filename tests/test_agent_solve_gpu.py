"""The per-thread solve kernel of large scenes on its rare paths (needs a GPU).

It keeps the nearest in registers by a network and puts equal distances in order
exactly.  Here: regular grids (every agent has ties), heaps of coincident agents
(more candidates at one distance than its list holds), routes, all compiled list
sizes, and the recorded active sets; bit for bit against the counting variant,
which keeps a sorted list, and against the warp-per-agent kernel.
"""
import numpy as np
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu

# agents, k, limits: the kernel's three list sizes, the last beyond 32 lines
SIZES = [(22500, 10, False), (22500, 7, True), (32400, 16, False), (1600, 30, True),
         (1600, 32, True)]


def _counted(ds):
    import torch
    ds.counters = torch.zeros(13, dtype=torch.int64, device="cuda")
    api.orca_scene_set_counters(ds.handle, ds.counters)
    return ds


def _both(s, n_steps=2):
    import torch
    got = []
    for counted in (False, True):
        ds = api.DeviceScene(s, "cuda", debug=True)
        if counted:
            _counted(ds)
        ds.step(n_steps)
        torch.cuda.synchronize()
        assert ds.sync_status() == 0
        got.append({"pos": ds.pos.clone(), "vel": ds.vel.clone(),
                    **{k: v.clone() for k, v in ds.dbg.items()}})
        if ds.wp_idx is not None:
            got[-1]["wp"] = ds.wp_idx.clone()
        ds.close()
    for k in got[0]:
        assert torch.equal(got[0][k], got[1][k]), k


def _limits(s, k, limits, seed):
    s.params.max_neighbors = k
    rng = np.random.default_rng(seed)
    if limits:
        s.type[rng.random(s.n) < 0.3] = 1
        s.params.vehicle_turn_rate, s.params.vehicle_accel = 0.8, 2.0
    return s


def _shuffled_grid(n, spacing, seed):
    m = int(round(n ** 0.5))
    s = scenes.open_square(m * m, spacing * m, seed=seed)
    g = np.stack(np.meshgrid(np.arange(m), np.arange(m)), -1).reshape(-1, 2)
    g = np.random.default_rng(seed).permutation(g)      # the index decides a tie
    s.pos = np.ascontiguousarray(spacing * (g + 0.5), dtype=np.float32)
    return s


@pytest.mark.parametrize("n,k,limits", SIZES)
@pytest.mark.parametrize("spacing", [0.75, 1.0, 1.3])
def test_regular_grids(n, k, limits, spacing):
    _both(_limits(_shuffled_grid(n, spacing, 100), k, limits, 1))


def _heaps(n, m, seed):
    s = scenes.open_square(n, (n / 0.4) ** 0.5, seed=seed)
    at = np.random.default_rng(seed).permutation(n) % max(1, n // m)
    s.pos = np.ascontiguousarray(s.pos[at])
    return s


@pytest.mark.parametrize("n,k,limits", SIZES)
@pytest.mark.parametrize("m", [3, 10, 40, 150, 800])
def test_heaps_of_coincident_agents(n, k, limits, m):
    _both(_limits(_heaps(n, m, 101), k, limits, 2), 1)


def test_heaps_cost_no_more_than_a_sorted_list():
    """A crowd let in at a few points: the list overflows again and again."""
    import torch
    s = _heaps(40000, 1000, 102)
    took = []
    for counted in (False, True):
        ds = api.DeviceScene(s)
        if counted:
            _counted(ds)
        pos = ds.pos.clone()
        best = 1e30
        for _ in range(4):
            ds.pos.copy_(pos)
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            ds.step(1)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        took.append(best)
        ds.close()
    assert took[0] <= 3.0 * took[1], took


def test_routes():
    s = scenes.waypoint_square(n_ped=19800, n_veh=300, side=220.0, seed=103)
    s.wp_idx[::3] = 1
    _both(s, 3)


def test_many_neighbours_above_the_warp_kernels_limit():
    s = scenes.open_square(132000, 575.0, seed=104)
    s.params.max_neighbors = 17
    _both(s, 1)


@pytest.mark.parametrize("n,k", [(16640, 10), (16641, 5), (19969, 12), (26625, 16), (47104, 17),
                                 (47105, 19), (57345, 20), (102401, 25), (122881, 27),
                                 (147457, 32)])
def test_around_the_limits(n, k):
    """On both sides of the sizes at which another solve kernel takes over."""
    s = scenes.open_square(n, (n / 0.5) ** 0.5, seed=107)
    s.params.max_neighbors = k
    rng = np.random.default_rng(5)
    s.vel = (0.5 * s.max_speed[:, None] * rng.standard_normal((s.n, 2))).astype(np.float32)
    _both(s, 1)


@pytest.mark.parametrize("grid", [False, True])
@pytest.mark.parametrize("n,k,limits", [(18000, 10, False), (18000, 10, True), (18000, 3, False),
                                        (28000, 14, True), (28000, 16, False),
                                        (46000, 17, False), (46000, 19, True)])
def test_recorded_active_sets(n, k, limits, grid):
    """The same 1,600 agents alone (a warp each) and with n more out of reach."""
    import torch
    s = _shuffled_grid(1600, 1.1, 105) if grid else scenes.open_square(1600, 50.0, seed=105)
    s = _limits(s, k, limits, 3)
    rng = np.random.default_rng(4)
    s.vel = (0.5 * s.max_speed[:, None] * rng.standard_normal((s.n, 2))).astype(np.float32)
    far = scenes.open_square(n, (n / 0.4) ** 0.5, seed=106)
    both = s.copy()
    for a in ("pos", "vel", "goal", "radius", "max_speed", "type"):
        x = getattr(far, a)
        if a in ("pos", "goal"):
            x = x + np.float32(500.0)
        setattr(both, a, np.ascontiguousarray(np.concatenate([getattr(s, a), x])))
    both.params.extent = (800.0, 800.0)
    acts = []
    for scene in (s, both):
        ds = api.DeviceScene(scene)
        ds.enable_debug(active=True)
        ds.step(2)
        torch.cuda.synchronize()
        assert ds.sync_status() == 0
        acts.append([ds.dbg["act"][:s.n].clone(), ds.dbg["nbr"][:s.n].clone(),
                     ds.vel[:s.n].clone()])
        ds.close()
    for a, b in zip(*acts):
        assert torch.equal(a, b)
