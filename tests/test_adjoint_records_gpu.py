"""The records that a rollout leaves for its adjoint (needs a GPU).

orca_rollout records its last segment, so the first orca_adjoint after it does
not replay that segment.  The gradient is the one that a replay gives (up to
the order of atomic sums, bound as in the checkpoint test): called again, after
another call on the same workspace, and with the rollout or the adjoint in a
CUDA graph; the forward results stay those of plain steps.
"""
import numpy as np
import pytest
import torch

from paper_2008_11578_gb300 import api, scenes
from paper_2008_11578_gb300.adjoint import Rollout

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-30))


@pytest.mark.parametrize("n_steps,every,k", [(6, 6, 10), (7, 3, 10), (5, 1, 10), (4, 8, 17)])
def test_recorded_segment_equals_its_replay(n_steps, every, k):
    s = scenes.waypoint_square(n_ped=700, n_veh=30, side=38.0, seed=96)
    s.params.max_neighbors = k
    g = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda *d: torch.randn(*d, device="cuda", generator=g)   # noqa: E731
    delta, gp, gv = 0.2 * rnd(n_steps, s.n, 2), rnd(s.n, 2), 0.1 * rnd(n_steps, s.n, 2)
    roll = Rollout(s, n_steps, every)

    def grads():
        return roll.backward_raw(delta, gp, gv, want_state0=True)

    def same(a, b):
        for x, y in zip(a, b):
            assert _rel(x, y) <= 1e-5

    roll.forward_raw(delta)
    pos, traj = roll.ds.pos.clone(), roll.vel_traj.clone()
    first = grads()
    same(grads(), first)                       # again, without a new rollout
    plain = api.DeviceScene(s, "cuda")
    for t in range(n_steps):
        plain.step(1, delta[t:t + 1].contiguous())
        assert torch.equal(plain.vel, traj[t])
    assert torch.equal(plain.pos, pos)

    # another call's records in the same workspace
    roll.forward_raw(delta)
    wp = torch.zeros(s.n, dtype=torch.uint8, device="cuda")
    out = [torch.empty((s.n, 2), device="cuda") for _ in range(2)]
    need = api.orca_adjoint_workspace_bytes(roll.ds.handle, 1, 1)
    if n_steps // every > 1:                   # (it leaves the first checkpoints alone)
        keep = roll.ws.clone()
        api.orca_step_vjp(roll.ds.handle, roll.ws, roll.ws_bytes, pos, traj[0], wp, None, gp, gp,
                          *out)
        assert need <= roll.ws_bytes
        roll.ws.copy_(keep)
        same(grads(), first)

    # in graphs: the rollout's, then the adjoint's twice for one rollout
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    dv = torch.empty((n_steps, s.n, 2), device="cuda")
    roll.reset()
    gr, ga = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr, stream=stream):
        api.orca_rollout(roll.ds.handle, n_steps, every, delta, roll.ws, roll.ws_bytes,
                         roll.vel_traj)
    with torch.cuda.graph(ga, stream=stream):
        api.orca_adjoint(roll.ds.handle, n_steps, every, delta, roll.ws, roll.ws_bytes, gp, gv, dv)
    roll.reset()
    gr.replay()
    torch.cuda.synchronize()
    assert torch.equal(roll.ds.pos, pos) and torch.equal(roll.vel_traj, traj)
    for _ in range(2):
        dv.zero_()
        ga.replay()
        torch.cuda.synchronize()
        assert _rel(dv, first[0]) <= 1e-5
    roll.close()
    plain.close()
