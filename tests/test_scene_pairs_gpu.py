"""Scenes side by side (needs a GPU): one made later, with smaller needs, takes
nothing from one made before."""
import pytest

from paper_2008_11578_gb300 import api, scenes

pytestmark = pytest.mark.gpu


def _scene(k, limits):
    s = scenes.shared_space(n_ped=180, n_veh=40, side=25.0, seed=98)
    s.params.max_neighbors = k
    if limits:
        s.params.vehicle_turn_rate, s.params.vehicle_accel = 0.8, 2.0
    return s


@pytest.mark.parametrize("kind", ["scene", "counting", "batch"])
@pytest.mark.parametrize("big,small", [((30, True), (32, False)), ((32, True), (25, True))])
def test_shared_memory_of_an_earlier_scene(big, small, kind):
    import torch

    def make(k, limits):
        if kind == "batch":
            return api.DeviceBatch([_scene(k, limits)])
        ds = api.DeviceScene(_scene(k, limits))
        if kind == "counting":
            ds.counters = torch.zeros(13, dtype=torch.int64, device="cuda")
            api.orca_scene_set_counters(ds.handle, ds.counters)
        return ds

    alone = make(*big)
    alone.step(2)
    first = make(*big)
    second = make(*small)
    first.step(2)
    second.step(1)
    torch.cuda.synchronize()
    assert first.sync_status() == 0 and second.sync_status() == 0
    assert torch.equal(first.pos, alone.pos) and torch.equal(first.vel, alone.vel)
    for x in (alone, first, second):
        x.close()
