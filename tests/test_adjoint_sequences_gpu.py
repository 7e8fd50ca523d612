"""The adjoint belongs to the checkpoints that are in its workspace (GPU).

Whatever ran before (calls, replayed CUDA graphs, another scene's calls, a
workspace put back from a copy), orca_adjoint gives the gradient of the rollout
whose checkpoints adj_ws holds.  Compared with a rollout and an adjoint of a
scene of their own, up to the order of the atomic sums (the bound of the
checkpoint test).
"""
import pytest
import torch

from paper_2008_11578_gb300 import api, scenes
from paper_2008_11578_gb300.adjoint import Rollout

pytestmark = pytest.mark.gpu

SEGMENTS = [(6, 6), (7, 3), (5, 1)]


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-30))


class _Case:
    def __init__(self, n_steps, every):
        self.s = scenes.waypoint_square(n_ped=500, n_veh=20, side=34.0, seed=97)
        self.steps, self.every = n_steps, every
        self.gen = torch.Generator(device="cuda").manual_seed(2)
        self.roll = Rollout(self.s, n_steps, every)
        self.offsets = [0.3 * self.rnd(n_steps, self.s.n, 2) for _ in range(2)]
        self.cots = [(self.rnd(self.s.n, 2), 0.1 * self.rnd(n_steps, self.s.n, 2))
                     for _ in range(2)]

    def rnd(self, *d):
        return torch.randn(*d, device="cuda", generator=self.gen)

    def adjoint(self, delta, cot, roll=None):
        return (roll or self.roll).backward_raw(delta, *cot, want_state0=True)

    def fresh(self, delta, cot):
        roll = Rollout(self.s, self.steps, self.every)
        roll.forward_raw(delta)
        out = [g.clone() for g in self.adjoint(delta, cot, roll)]
        roll.close()
        return out

    def check(self, got, delta, cot):
        for a, b in zip(got, self.fresh(delta, cot)):
            assert _rel(a, b) <= 1e-5

    def rollout(self, delta):
        api.orca_rollout(self.roll.ds.handle, self.steps, self.every, delta, self.roll.ws,
                         self.roll.ws_bytes, self.roll.vel_traj)


def _capture(fn):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        fn()
    return graph


@pytest.mark.parametrize("n_steps,every", SEGMENTS)
def test_rollout_graph_replayed_after_a_plain_rollout(n_steps, every):
    c = _Case(n_steps, every)
    delta = c.offsets[0].clone()
    c.roll.reset()
    graph = _capture(lambda: c.rollout(delta))
    c.roll.forward_raw(delta)
    delta.copy_(c.offsets[1])
    c.roll.reset()
    graph.replay()
    for cot in c.cots:                       # the first gradient, and one after it
        c.check(c.adjoint(delta, cot), delta, cot)
    c.roll.close()


@pytest.mark.parametrize("n_steps,every", SEGMENTS)
def test_adjoint_graph_replayed_between_rollout_and_adjoint(n_steps, every):
    c = _Case(n_steps, every)
    delta, dv = c.offsets[0], torch.empty_like(c.offsets[0])
    c.roll.forward_raw(delta)
    graph = _capture(lambda: api.orca_adjoint(
        c.roll.ds.handle, n_steps, every, delta, c.roll.ws, c.roll.ws_bytes, *c.cots[0], dv))
    c.roll.forward_raw(delta)
    graph.replay()
    torch.cuda.synchronize()
    assert _rel(dv, c.fresh(delta, c.cots[0])[0]) <= 1e-5
    c.check(c.adjoint(delta, c.cots[1]), delta, c.cots[1])
    c.roll.close()


@pytest.mark.parametrize("n_steps,every", SEGMENTS)
def test_workspace_put_back_from_a_copy(n_steps, every):
    c = _Case(n_steps, every)
    c.roll.forward_raw(c.offsets[0])
    c.adjoint(c.offsets[0], c.cots[0])
    keep = c.roll.ws.clone()
    c.roll.forward_raw(c.offsets[1])
    c.roll.ws.copy_(keep)
    c.check(c.adjoint(c.offsets[0], c.cots[1]), c.offsets[0], c.cots[1])
    c.roll.close()


def test_single_step_products_between_rollout_and_adjoint():
    """A VJP leaves the checkpoint of a one-segment rollout alone, whether this
    scene or another one calls it."""
    c = _Case(6, 6)
    other = api.DeviceScene(c.s)
    out = [torch.empty((c.s.n, 2), device="cuda") for _ in range(2)]
    wp = torch.zeros(c.s.n, dtype=torch.uint8, device="cuda")
    for handle in (c.roll.ds.handle, other.handle):
        c.roll.forward_raw(c.offsets[0])
        api.orca_step_vjp(handle, c.roll.ws, c.roll.ws_bytes, c.roll.ds.pos.clone(),
                          c.roll.vel_traj[0].contiguous(), wp, None, *c.cots[0][:1],
                          c.cots[1][0], *out)
        c.check(c.adjoint(c.offsets[0], c.cots[1]), c.offsets[0], c.cots[1])
    other.close()
    c.roll.close()
