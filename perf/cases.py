"""The work a user of this package has it do, as a list of measurable cases.

A case is a crowd of one of the families of ``scenes.py`` (or a batch of
them), a number of steps, and how the steps are run: plain calls, a recorded
CUDA graph, a differentiable rollout with its gradient, or a step followed by
the removal of arrived agents.  Every pass starts from the same state (the
crowd in motion), so passes are alike; the state is put back with a
device-to-device copy, as a program does that evaluates a scenario again.
"""
import math

import numpy as np
import torch

from paper_2008_11578_gb300 import api, scenes
from paper_2008_11578_gb300.adjoint import Rollout

# kinds of crowd, and the sizes drawn for each
SQUARE_DENSITY = 0.4        # agents per m^2 of the 1,000-agent open square (50 m)
CLUSTER_AGENTS = 15625      # agents per Gaussian cluster of the 1M workload


def listed():
    return [
        # one frame of a small plaza: the smallest call, an interactive loop
        dict(name="frame_1k", kind="square", n=1000, steps=1),
        # the same plaza run ahead several steps in one call
        dict(name="run_1k", kind="square", n=1000, steps=10),
        # a mid-sized square whose agents see the most neighbours allowed
        dict(name="wide_8k", kind="square", n=8191, steps=2, k=32),
        # shared space: pedestrian streams crossing vehicle lanes whose
        # vehicles have turn-rate and acceleration limits, several steps
        dict(name="limits_16k", kind="crossing", n=16250, steps=4, limits=True),
        # one frame of the paper-sized shared space
        dict(name="crossing_65k", kind="crossing", n=65000, steps=1),
        # dense clusters over several steps of one call
        dict(name="clusters_250k", kind="clusters", n=250000, steps=4),
        # one frame of the million-agent stress scene, the headline workload, with
        # the cell size that the autotuner picks for it
        dict(name="clusters_1m", kind="clusters", n=1000000, steps=1, cell=2.0),
        # a handful of small scenes replayed from a CUDA graph (data generation
        # and policy evaluation loops)
        dict(name="batch_48", kind="batch", n_scenes=48, lo=100, hi=1000, steps=4, graph=True),
        # many scenes of uneven size, the largest amount of work
        dict(name="batch_512", kind="batch", n_scenes=512, lo=100, hi=20000, steps=2),
        # trajectory optimisation: a differentiable rollout and its gradient
        dict(name="gradient_4k", kind="gradient", n=4064, steps=16, every=8),
        # an evacuation loop: one step, then whoever is at the goal leaves (here
        # nobody is there yet, as in most frames, so a pass can be repeated)
        dict(name="evacuation_100k", kind="evacuation", n=99999, steps=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["square", "square", "crossing", "clusters", "batch", "gradient",
                       "evacuation"])
    if kind == "square":
        return dict(kind=kind, n=_log_int(rng, 150, 30000), steps=rng.randint(1, 8),
                    k=rng.choice([5, 10, 10, 10, 16, 17, 32]), graph=rng.random() < 0.3)
    if kind == "crossing":
        return dict(kind=kind, n=_log_int(rng, 2000, 150000), steps=rng.randint(1, 4),
                    limits=rng.random() < 0.4)
    if kind == "clusters":
        return dict(kind=kind, n=_log_int(rng, 60000, 1000000), steps=rng.randint(1, 2),
                    cell=rng.choice([1.0, 1.5, 2.0]))
    if kind == "batch":
        return dict(kind=kind, n_scenes=_log_int(rng, 8, 400), lo=100,
                    hi=_log_int(rng, 500, 15000), steps=rng.randint(1, 3),
                    graph=rng.random() < 0.5)
    if kind == "gradient":
        return dict(kind=kind, n=_log_int(rng, 500, 9000), steps=rng.randint(4, 16),
                    every=rng.randint(2, 8))
    return dict(kind=kind, n=_log_int(rng, 10000, 300000), steps=1)


# ----------------------------------------------------------------- inputs ----

def _in_motion(s, rng):
    """Agents under way: toward the goal at most of their speed, with noise."""
    d = s.goal - s.pos
    d /= np.maximum(np.linalg.norm(d, axis=1, keepdims=True), 1e-6)
    speed = s.max_speed[:, None] * rng.uniform(0.5, 1.0, (s.n, 1))
    v = d * speed + 0.1 * s.max_speed[:, None] * rng.standard_normal((s.n, 2))
    v *= np.minimum(1.0, s.max_speed[:, None] / np.maximum(np.linalg.norm(v, axis=1,
                                                                          keepdims=True), 1e-6))
    s.vel = np.ascontiguousarray(v, dtype=np.float32)
    return s


def _scenes(case, seed):
    """The case's scenes (one, or the batch's), made from the seed alone."""
    rng = np.random.default_rng([seed, 77])
    kind, n = case["kind"], case.get("n", 0)
    if kind == "batch":
        sizes = scenes.batched_sizes(case["n_scenes"], case["lo"], case["hi"])
        return [_in_motion(scenes.batched(1, m, m, seed=[seed, i])[0], rng)
                for i, m in enumerate(sizes)]
    if kind == "square":
        s = scenes.open_square(n, math.sqrt(n / SQUARE_DENSITY), seed=seed)
        s.params.max_neighbors = case.get("k", 10)
    elif kind == "gradient":
        n_veh = max(1, n // 64)
        s = scenes.waypoint_square(n - n_veh, n_veh, math.sqrt(n / 0.4064), seed=seed)
    elif kind == "clusters":
        a = max(1, int(round(math.sqrt(n / CLUSTER_AGENTS))))
        s = scenes.clusters(n, 250.0 * a, a, seed=seed)
    else:
        n_veh = n // 65 if kind == "crossing" else 0
        s = scenes.shared_space(n - n_veh, n_veh, 500.0 * math.sqrt(n / 65000.0), seed=seed)
        if case.get("limits"):
            s.params.vehicle_turn_rate, s.params.vehicle_accel = 0.8, 2.0
    return [_in_motion(s, rng)]


def _cotangents(case, seed, n):
    g = np.random.default_rng([seed, 78])
    t = case["steps"]
    return (g.normal(0, 0.2, (t, n, 2)).astype(np.float32),
            g.normal(0, 1.0, (n, 2)).astype(np.float32),
            g.normal(0, 0.1, (t, n, 2)).astype(np.float32))


def prepare(case, seed):
    sl = _scenes(case, seed)
    kind = case["kind"]
    if kind == "gradient":
        s = sl[0]
        delta, gp, gv = (torch.as_tensor(a, device="cuda") for a in _cotangents(case, seed, s.n))
        return dict(case=case, roll=Rollout(s, case["steps"], case["every"]),
                    delta=delta.requires_grad_(True),
                    way=torch.as_tensor(s.waypoints, device="cuda").requires_grad_(True),
                    gp=gp, gv=gv)
    if kind == "batch":
        dev = api.DeviceBatch(sl)
    else:
        dev = api.DeviceScene(sl[0], cell_size=case.get("cell"))
    if case.get("graph"):
        dev.capture(case["steps"])
    return dict(case=case, dev=dev, pos=dev.pos.clone(), vel=dev.vel.clone())


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        pos, vel = state["roll"](state["delta"], state["way"])
        gd, gw = torch.autograd.grad([pos, vel], [state["delta"], state["way"]],
                                     [state["gp"], state["gv"]])
        return dict(pos=pos.detach(), vel=vel.detach(), grad_delta=gd, grad_way=gw)
    dev = state["dev"]
    dev.pos.copy_(state["pos"])
    dev.vel.copy_(state["vel"])
    if case.get("graph"):
        dev.replay()
    else:
        dev.step(case["steps"])
    out = dict(pos=dev.pos, vel=dev.vel)
    if case["kind"] == "evacuation":
        out["kept"] = dev.remove_arrived()
    return out


# ------------------------------------------------------------------- work ----

def _agents(case):
    if case["kind"] != "batch":
        return case["n"]
    lo, hi = case["lo"], case["hi"]
    return case["n_scenes"] * (hi - lo) / math.log(hi / lo)   # mean of the log-uniform sizes


def work(case):
    """State and agent constants in, new state out (each once per pass); per
    agent and step the k neighbours' keys and half-planes (60 flops) and a
    linear program that tests each once more (10 flops)."""
    n, k, t = _agents(case), case.get("k", 10), case["steps"]
    per_agent = 16 + 8 + 4 + 4 + 1 + 16
    flops = n * t * k * (6 + 60 + 10)
    if case["kind"] == "gradient":   # offsets in; velocities, both cotangents and gradients
        return dict(bytes=n * (per_agent + 8 + t * 8 * 4), flops=2 * flops)
    if case["kind"] == "evacuation":
        per_agent += 4
    return dict(bytes=n * per_agent, flops=flops)


# ------------------------------------------------------------------ exact ----
# The step in 64 bits: neighbours by the 32-bit keys that define them, every
# line and linear program in double precision, the programs by enumeration of
# the points where an optimum can lie.

def _neighbours(p32, cellpos, r_n, k):
    """Indices [n, k] of the k nearest within r_n by (32-bit d^2, index), -1 padded."""
    n = p32.shape[0]
    out = torch.full((n, k), -1, dtype=torch.long, device=p32.device)
    todo = torch.arange(n, device=p32.device)
    r2 = torch.tensor(r_n, dtype=torch.float32) ** 2
    h = min(2.0, r_n)
    big = torch.iinfo(torch.int64).max
    while todo.numel():
        lo = cellpos.min(0).values
        c = ((cellpos - lo) / h).floor().long() + 1
        nx = int(c[:, 0].max()) + 2
        cid = c[:, 1] * nx + c[:, 0]
        order = torch.argsort(cid)
        sid = cid[order].contiguous()
        again = []
        at = 0
        while at < todo.numel():
            q = todo[at:at + 200000]
            rows = torch.stack([cid[q] + d * nx for d in (-1, 0, 1)], 1)
            b = torch.searchsorted(sid, (rows - 1).contiguous())
            e = torch.searchsorted(sid, (rows + 1).contiguous(), right=True)
            length = int((e - b).max())
            m = max(1, min(q.numel(), 60_000_000 // (3 * max(length, 1))))
            q, b, e = q[:m], b[:m], e[:m]
            at += m
            j = b[:, :, None] + torch.arange(length, device=q.device)
            ok = (j < e[:, :, None]).reshape(m, -1)
            j = order[j.clamp_max(n - 1)].reshape(m, -1)
            d = p32[j] - p32[q][:, None]
            dd = d * d
            d2 = dd[..., 0] + dd[..., 1]
            ok &= (d2 < r2) & (j != q[:, None])
            key = torch.where(ok, (d2.view(torch.int32).long() << 32) | j, big)
            kk = min(k, key.shape[1])
            best = key.topk(kk, dim=1, largest=False, sorted=True).values
            idx = torch.where(best == big, -1, best & 0xffffffff)
            far = torch.where(best[:, -1] == big, math.inf,
                              (best[:, -1] >> 32).int().view(torch.float32).double())
            done = (far < (0.999 * h) ** 2) & (kk == k) | (h >= r_n)
            out[q, :kk] = torch.where(done[:, None], idx, out[q, :kk])
            again.append(q[~done])
        todo = torch.cat(again)
        h = r_n if 2 * h > r_n else 2 * h
    return out


def _det(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _lines(p, v, rad, typ, nbr, par):
    """Half-planes (point, direction, valid) [n, k(+3)] of every agent."""
    ok = nbr >= 0
    j = nbr.clamp_min(0)
    r32 = rad[:, None] + rad[j]
    d32 = p.float()[j] - p.float()[:, None]
    d32 = d32 * d32
    over = (d32[..., 0] + d32[..., 1]) <= r32 * r32
    q, w = p[j] - p[:, None], v[:, None] - v[j]
    rho = rad.double()[:, None] + rad.double()[j]
    ft = torch.as_tensor(np.asarray(par.f, np.float32), device=p.device).double()
    f = ft[typ.long()[:, None], typ.long()[j]][..., None]
    t = torch.where(over, 1.0 / par.dt, 1.0 / par.time_horizon)
    wc = w - q * t[..., None]
    wq, ww = (wc * q).sum(-1), (wc * wc).sum(-1)
    cap = over | ((wq < 0) & (wq * wq > rho * rho * ww))
    hc = wc / ww.sqrt().clamp_min(1e-300)[..., None]
    u_cap = (rho * t - ww.sqrt())[..., None] * hc
    d_cap = torch.stack([hc[..., 1], -hc[..., 0]], -1)
    qq = (q * q).sum(-1).clamp_min(1e-300)
    leg = (qq - rho * rho).clamp_min(0).sqrt()
    s = torch.where(_det(q, w) > 0, 1.0, -1.0)
    d_leg = torch.stack([s * q[..., 0] * leg - q[..., 1] * rho,
                         q[..., 0] * rho + s * q[..., 1] * leg], -1) / qq[..., None]
    u_leg = (w * d_leg).sum(-1, keepdim=True) * d_leg - w
    d = torch.where(cap[..., None], d_cap, d_leg)
    pt = v[:, None] + f * torch.where(cap[..., None], u_cap, u_leg)
    return pt, d, ok


def _limit_lines(v, vp, typ, par):
    """The vehicles' turn-rate and acceleration half-planes [n, 3]."""
    sp = v.norm(dim=1)
    moving = sp * sp >= 0.01
    pl = vp.norm(dim=1)
    h = torch.where(moving[:, None], v / sp.clamp_min(1e-300)[:, None],
                    vp / pl.clamp_min(1e-300)[:, None])
    th = par.vehicle_turn_rate * par.dt
    c, s = math.cos(th), math.sin(th)
    left = torch.stack([c * h[:, 0] - s * h[:, 1], s * h[:, 0] + c * h[:, 1]], -1)
    right = torch.stack([c * h[:, 0] + s * h[:, 1], -s * h[:, 0] + c * h[:, 1]], -1)
    top = torch.where(moving, sp, 0.0) + par.vehicle_accel * par.dt
    zero = torch.zeros_like(v)
    d = torch.stack([-left, right, torch.stack([-h[:, 1], h[:, 0]], -1)], 1)
    pt = torch.stack([zero, zero, top[:, None] * h], 1)
    veh = typ != 0
    return pt, d, torch.stack([veh & moving, veh & moving, veh & (moving | (pl > 0))], 1)


def _rim(pt, d, vmax):
    """Both points of lines pt + s d (unit d) on the circle |v| = vmax; NaN where it misses."""
    dot = (pt * d).sum(-1)
    sq = (dot * dot + (vmax * vmax)[:, None] - (pt * pt).sum(-1)).sqrt()
    return torch.cat([pt + (-dot - sq)[..., None] * d, pt + (-dot + sq)[..., None] * d], 1)


def _programs(pt, d, ok, vmax, vp):
    """The admissible velocity nearest vp, else that of least penetration."""
    n, m = ok.shape
    dev = pt.device
    nrm = torch.stack([-d[..., 1], d[..., 0]], -1)
    c = _det(d, pt)
    low = torch.where(ok, 0.0, -math.inf)

    def worst(x):   # [n, q, 2] -> largest penetration of each candidate
        t = torch.full(x.shape[:2], -math.inf, dtype=x.dtype, device=dev)
        for i in range(m):
            t = torch.maximum(t, c[:, i, None] - (x * nrm[:, i, None]).sum(-1) + low[:, i, None])
        return t

    i2 = torch.combinations(torch.arange(m, device=dev), 2)
    ok2 = ok[:, i2].all(-1)
    inside = lambda x: x.norm(dim=-1) <= vmax[:, None] * (1 + 1e-12) + 1e-13   # noqa: E731

    def least(cands, valid, best_t, best_v):
        t = torch.where(valid & inside(cands), worst(cands), math.inf)
        t = torch.where(t.isnan(), math.inf, t)
        bt, bi = t.min(1)
        bv = cands.gather(1, bi[:, None, None].expand(-1, 1, 2))[:, 0]
        win = bt < best_t
        return torch.where(win, bt, best_t), torch.where(win[:, None], bv, best_v)

    best_t = torch.full((n,), math.inf, dtype=pt.dtype, device=dev)
    best_v = torch.zeros_like(vp)
    best_t, best_v = least(vmax[:, None, None] * nrm, ok, best_t, best_v)
    if m > 1:
        a = nrm[:, i2[:, 1]] - nrm[:, i2[:, 0]]       # planes i and j penetrate alike on a . v = b
        b = c[:, i2[:, 1]] - c[:, i2[:, 0]]
        a2 = (a * a).sum(-1)
        base = a * (b / a2)[..., None]
        e = torch.stack([a[..., 1], -a[..., 0]], -1) / a2.sqrt()[..., None]
        best_t, best_v = least(_rim(base, e, vmax), torch.cat([ok2, ok2], 1), best_t, best_v)
    i3 = torch.combinations(torch.arange(m, device=dev), 3)
    for at in range(0, i3.shape[0], 256):
        i, j, l = i3[at:at + 256].unbind(1)
        a, g = nrm[:, j] - nrm[:, i], nrm[:, l] - nrm[:, i]
        x, y = c[:, j] - c[:, i], c[:, l] - c[:, i]
        det = _det(a, g)
        cand = torch.stack([x * g[..., 1] - y * a[..., 1],
                            a[..., 0] * y - g[..., 0] * x], -1) / det[..., None]
        best_t, best_v = least(cand, ok[:, i] & ok[:, j] & ok[:, l], best_t, best_v)

    # admissible candidates: vp (capped), on each line, crossings, line ends on the rim
    speed = vp.norm(dim=1, keepdim=True)
    cands = [torch.where(speed > vmax[:, None], vp * (vmax[:, None] / speed.clamp_min(1e-300)),
                         vp)[:, None],
             pt + ((vp[:, None] - pt) * d).sum(-1, keepdim=True) * d, _rim(pt, d, vmax)]
    valid = [torch.ones((n, 1), dtype=torch.bool, device=dev), ok, ok, ok]
    if m > 1:
        li, lj = i2.unbind(1)
        s = _det(d[:, lj], pt[:, li] - pt[:, lj]) / _det(d[:, li], d[:, lj])
        cands.append(pt[:, li] + s[..., None] * d[:, li])
        valid.append(ok2)
    cands, valid = torch.cat(cands, 1), torch.cat(valid, 1)
    good = valid & inside(cands) & (worst(cands) <= 1e-10)
    dist = torch.where(good, (cands - vp[:, None]).norm(dim=-1), math.inf)
    near, at = dist.nan_to_num(math.inf, math.inf).min(1)
    v2 = cands.gather(1, at[:, None, None].expand(-1, 1, 2))[:, 0]
    return torch.where((near < math.inf)[:, None], v2, best_v)


def _exact_step(p, v, wp, s, delta):
    """One step of the crowd ``s`` (tensors) from the 64-bit state p, v."""
    par = s["par"]
    goal = s["goal"].double()
    if wp is not None:
        on = s["route"] >= 0
        table = s["way"].double()[s["route"].clamp_min(0).long()]
        target = table.gather(1, wp[:, None, None].expand(-1, 1, 2))[:, 0]
        hit = ((target - p) ** 2).sum(1) <= s["rad"].double() ** 2
        wp = torch.where(on & hit & (wp < table.shape[1] - 1), wp + 1, wp)
        target = table.gather(1, wp[:, None, None].expand(-1, 1, 2))[:, 0]
        goal = torch.where(on[:, None], target, goal)
    g = goal - p
    gl = g.norm(dim=1)
    vmax = s["vmax"].double()
    vp = g * torch.minimum(vmax / gl.clamp_min(1e-300), torch.full_like(gl, 1 / par.dt))[:, None]
    if delta is not None:
        vp = vp + delta
    nbr = _neighbours(p.float(), p + s["shift"], par.neighbor_dist, par.max_neighbors)
    vn = torch.empty_like(v)
    m = par.max_neighbors + 3
    size = 600_000 // m          # agents at a time: a few GB of candidates
    pts, ds, oks = _lines(p, v, s["rad"], s["typ"], nbr, par)
    if par.vehicle_turn_rate > 0:
        pts, ds, oks = (torch.cat([a, b], 1) for a, b in
                        zip((pts, ds, oks), _limit_lines(v, vp, s["typ"], par)))
    for at in range(0, p.shape[0], size):
        o = slice(at, at + size)
        vn[o] = _programs(pts[o], ds[o], oks[o], vmax[o], vp[o])
    return p + par.dt * vn, vn, wp


def exact(case, seed):
    sl = _scenes(case, seed)

    def cat(get, dt=None):
        return torch.as_tensor(np.concatenate([get(s) for s in sl]), device="cuda", dtype=dt)

    # scenes of a batch do not see each other: 100 m between them when searching
    wide = np.cumsum([0.0] + [s.params.extent[0] + 100.0 for s in sl])
    shift = np.concatenate([np.full(s.n, x) for s, x in zip(sl, wide)])
    t = dict(par=sl[0].params, goal=cat(lambda s: s.goal), rad=cat(lambda s: s.radius),
             vmax=cat(lambda s: s.max_speed), typ=cat(lambda s: s.type),
             shift=torch.as_tensor(np.stack([shift, 0 * shift], 1), device="cuda"))
    p, v = cat(lambda s: s.pos).double(), cat(lambda s: s.vel).double()
    wp = delta = None
    if case["kind"] == "gradient":
        s = sl[0]
        t["route"] = torch.as_tensor(s.route, device="cuda")
        t["way"] = torch.as_tensor(s.waypoints, device="cuda")
        wp = torch.as_tensor(s.wp_idx, device="cuda").long()
        delta = torch.as_tensor(_cotangents(case, seed, s.n)[0], device="cuda").double()
    vels = []
    for i in range(case["steps"]):
        p, v, wp = _exact_step(p, v, wp, t, None if delta is None else delta[i])
        vels.append(v)
    if case["kind"] == "gradient":
        # the gradient holds every discrete choice of the 32-bit trajectory fixed
        return dict(pos=p, vel=torch.stack(vels), grad_delta=None, grad_way=None)
    out = dict(pos=p, vel=v)
    if case["kind"] == "evacuation":
        out["kept"] = None
    return out
