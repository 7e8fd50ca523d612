"""Steps of scenes with numbers that are none, or beyond all measure (GPU).

The call reports a non-finite position or velocity; the other agents' results
are those of the same scene in the counting variant (one thread per agent, a
sorted list, one loop over the lines), whichever kernel solves the step.
"""
import numpy as np
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu

# agents, k, limits: a warp per agent (without cells, with cells), the register
# network's three sizes, the sorted list
SIZES = [(900, 10, False), (3000, 10, False), (3000, 14, True), (2000, 32, False),
         (18000, 10, False), (18000, 7, True), (28000, 16, False), (1500, 32, True),
         (48000, 17, False)]


def _scene(n, k, limits):
    s = scenes.shared_space(n_ped=n - n // 10, n_veh=n // 10, side=(n / 0.45) ** 0.5, seed=108)
    g = np.random.default_rng(6)
    s.vel = (0.6 * s.max_speed[:, None] * g.standard_normal((n, 2))).astype(np.float32)
    s.params.max_neighbors = k
    if limits:
        s.params.vehicle_turn_rate, s.params.vehicle_accel = 0.8, 2.0
    return s


def _same(a, b):
    return a.shape == b.shape and np.array_equal(a, b, equal_nan=a.dtype.kind == "f")


def _both(s, status, delta=None):
    import torch
    got = []
    for counted in (False, True):
        ds = api.DeviceScene(s, "cuda", debug=True)
        if counted:
            counters = torch.zeros(13, dtype=torch.int64, device="cuda")
            api.orca_scene_set_counters(ds.handle, counters)
        ds.step(1, delta)
        torch.cuda.synchronize()
        assert ds.sync_status() == status
        got.append({"pos": ds.pos.cpu().numpy(), "vel": ds.vel.cpu().numpy(),
                    **{k: v.cpu().numpy() for k, v in ds.dbg.items()}})
        ds.close()
    for k in got[0]:
        assert _same(got[0][k], got[1][k]), k


@pytest.mark.parametrize("n,k,limits", SIZES)
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_positions(n, k, limits, axis, value):
    s = _scene(n, k, limits)
    s.pos[::37, axis] = value
    _both(s, 4)


@pytest.mark.parametrize("n,k,limits", SIZES)
@pytest.mark.parametrize("field,value", [("vel", 1e13), ("vel", 1e19), ("vel", 3e38),
                                         ("vel", np.nan), ("radius", np.nan), ("radius", np.inf),
                                         ("radius", -1.0), ("max_speed", -5.0),
                                         ("max_speed", np.inf), ("max_speed", np.nan),
                                         ("goal", np.inf), ("dt", 1e-20), ("dt", 1e-39)])
def test_half_planes(n, k, limits, field, value):
    """Half-planes whose products overflow, or that are no numbers."""
    s = _scene(n, k, limits)
    with np.errstate(all="ignore"):
        if field == "dt":
            s.params.dt = value
        elif field == "vel":
            s.vel[::41] *= np.float32(value)
        else:
            getattr(s, field)[::41] = value
    bad = not np.isfinite(s.vel).all()
    _both(s, 4 if bad else 0)
