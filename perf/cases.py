"""What a user has the fleet simulator do, as cases that can be timed and compared.

Six kinds of work, each through the package's public entry points:

  reach    one step of ReachEnv, as a policy-training loop takes it: actions in; observations,
           rewards, done and collision flags out (episodes that end are re-drawn inside the step)
  control  one control period of a Fleet among obstacles: new targets in, one step, states out
  rollout  a Fleet set to given states and run for many steps (evaluation, sampling-based planning),
           optionally with a masked reset first
  depth    one depth image per camera against the environments' boxes
  adjoint  one training iteration of the differentiable rollout: loss, and its gradients
  serve    a batch of requests through the continuous-batching server, from submit to results

`exact` computes the same in 64 bits with plain torch, written from the equations: the SE(3) controller
in its three modes, allocation with clamp and motor lag, semi-implicit Euler or RK4, the sphere-vs-box
test, the Philox reset draw, the pinhole slab caster, and autograd for the gradients.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2305_16510_gb300 import _abi
from paper_2305_16510_gb300.autograd import rollout_loss
from paper_2305_16510_gb300.fleet import Fleet
from paper_2305_16510_gb300.serving import RequestPool, Server
from paper_2305_16510_gb300.task import ReachEnv

MODES = {"pos": (0,), "vel": (1,), "att": (2,), "att_vel": (1, 2), "all": (0, 1, 2)}


# ------------------------------------------------------------------ the cases --
def listed():
    return [
        # a small policy-training batch on attitude commands: every step is one short call, so launches
        # and latency are what it costs
        dict(name="reach_small", kind="reach", n=4096, modes="att", integrator=0, substeps=1, n_obs=0, airframes="quad"),
        # the largest training batch: a million environments, one pass over their state per step
        dict(name="reach_large", kind="reach", n=1 << 20, modes="att", integrator=0, substeps=1, n_obs=0,
             airframes="quad"),
        # navigation training among 16 re-placed boxes on velocity commands, RK4 at 2.5 ms
        dict(name="reach_boxes", kind="reach", n=131072, modes="vel", integrator=1, substeps=4, n_obs=16,
             airframes="quad"),
        # an outer-loop controller over an obstacle fleet of ragged size: targets in, one step, states out
        dict(name="control_boxes", kind="control", n=250007, modes="all", integrator=1, substeps=4, n_obs=16,
             airframes="quad"),
        # the million-quad obstacle rollout of the benchmark, one call of 1,000 steps
        dict(name="rollout_boxes", kind="rollout", n=1 << 20, steps=1000, modes="all", integrator=1, substeps=4,
             n_obs=16, airframes="quad", drag=0.0, masked=False),
        # the paper's throughput fleet: 131,072 quads on attitude or velocity commands, no obstacles
        dict(name="rollout_paper", kind="rollout", n=131072, steps=100, modes="att_vel", integrator=0, substeps=1,
             n_obs=0, airframes="quad", drag=0.0, masked=False),
        # four million quads, hexas and octos with drag, 1 % of them reset, then 50 steps
        dict(name="rollout_mixed", kind="rollout", n=4194304, steps=50, modes="vel", integrator=0, substeps=1, n_obs=0,
             airframes="mixed", drag=0.1, masked=True),
        # depth images of 1,024 vehicles at the paper's camera resolution
        dict(name="depth_large", kind="depth", n=1024, cams=1024, width=480, height=270, n_obs=16, hfov=1.5184,
             max_range=10.0, offset=False),
        # a few cameras of chosen vehicles, odd image size, camera mounted off the centre
        dict(name="depth_small", kind="depth", n=512, cams=61, width=213, height=117, n_obs=13, hfov=1.2,
             max_range=8.0, offset=True),
        # gradient of a 256-step tracking loss for 65,536 vehicles, w.r.t. initial states and gains
        dict(name="adjoint_large", kind="adjoint", n=65536, steps=256, modes="pos", targets_grad=False),
        # a small ragged batch learning its velocity and attitude commands through the controller
        dict(name="adjoint_small", kind="adjoint", n=1000, steps=256, modes="att_vel", targets_grad=True),
        # eight rollout requests of mixed size, horizon and box count, submitted together
        dict(name="serve_batch", kind="serve", requests=8, n=4096, steps=200, substeps=4, integrator=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (sizes log-uniform, mostly odd)."""
    kind = rng.choice(("reach", "reach", "control", "rollout", "rollout", "depth", "adjoint", "serve"))
    integrator = rng.choice((0, 1))
    substeps = rng.choice((1, 2, 4))
    n_obs = rng.choice((0, rng.randint(1, 32)))
    if kind == "reach":
        return dict(kind=kind, n=_log_int(rng, 500, (1 << 20) if n_obs == 0 else (1 << 18)),
                    modes=rng.choice(("att", "vel")), integrator=integrator, substeps=substeps, n_obs=n_obs,
                    airframes=rng.choice(("quad", "quad", "mixed")))
    if kind == "control":
        return dict(kind=kind, n=_log_int(rng, 500, 1 << 18), modes=rng.choice(tuple(MODES)), integrator=integrator,
                    substeps=substeps, n_obs=rng.randint(1, 32), airframes=rng.choice(("quad", "quad", "mixed")))
    if kind == "rollout":
        steps = _log_int(rng, 2, 1000)
        top = min(1 << 20, (1 << 28) // (steps * substeps))
        return dict(kind=kind, n=_log_int(rng, 500, top), steps=steps, modes=rng.choice(tuple(MODES)),
                    integrator=integrator, substeps=substeps, n_obs=n_obs, airframes=rng.choice(("quad", "mixed")),
                    drag=rng.choice((0.0, 0.1)), masked=rng.random() < 0.3)
    if kind == "depth":
        width, height = rng.randint(32, 640), rng.randint(24, 480)
        cams = _log_int(rng, 1, min(1024, (1 << 27) // (width * height)))
        return dict(kind=kind, n=max(cams, 512), cams=cams, width=width, height=height, n_obs=rng.randint(1, 32),
                    hfov=round(rng.uniform(0.9, 1.9), 3), max_range=rng.choice((5.0, 10.0, 20.0)),
                    offset=rng.random() < 0.5)
    if kind == "adjoint":
        steps = _log_int(rng, 16, 300)
        return dict(kind=kind, n=_log_int(rng, 200, (1 << 24) // steps), steps=steps, modes=rng.choice(tuple(MODES)),
                    targets_grad=rng.random() < 0.5)
    return dict(kind=kind, requests=rng.randint(1, 16), n=_log_int(rng, 300, 16384), steps=rng.randint(50, 400),
                substeps=substeps, integrator=integrator)


# ------------------------------------------------------------------ the inputs --
def _split(n, airframes):
    """(quads, hexas, octos), in contiguous ranges."""
    if airframes == "quad":
        return n, 0, 0
    hexa, octo = int(round(0.4 * n)), int(round(0.2 * n))
    return n - hexa - octo, hexa, octo


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float32)


def _quat(angle, axis):
    half = 0.5 * angle
    return torch.cat((torch.cos(half)[None], torch.sin(half) * axis / axis.norm(dim=0, keepdim=True)))


def _commands(g, n, modes, mass):
    """Modes uint8 [n] and each mode's targets float32 [4, n]."""
    mix = torch.tensor(MODES[modes], device="cuda", dtype=torch.uint8)
    md = mix[torch.randint(len(mix), (n,), generator=g, device="cuda")]
    pos = torch.cat((_uniform(g, -3, 3, 3, n), _uniform(g, -math.pi, math.pi, 1, n)))
    vel = torch.cat((_uniform(g, -2, 2, 3, n), _uniform(g, -1, 1, 1, n)))
    a30 = math.radians(30)
    att = torch.cat((_uniform(g, -a30, a30, 2, n), _uniform(g, -1, 1, 1, n),
                     _uniform(g, 0.5, 1.5, 1, n) * (mass * 9.81)[None]))
    return md, torch.where(md == 0, pos, torch.where(md == 1, vel, att)).contiguous()


def _boxes(g, n_obs, n):
    """float32 [n_obs, 10, n]: centres U[-5, 5]^3, half-extents U[0.1, 1], orientation uniform on SO(3)."""
    b = torch.empty((n_obs, 10, n), device="cuda")
    for k in range(n_obs):
        b[k, 0:3] = _uniform(g, -5, 5, 3, n)
        b[k, 3:6] = _uniform(g, 0.1, 1.0, 3, n)
        u = torch.randn((4, n), generator=g, device="cuda")
        b[k, 6:10] = u / u.norm(dim=0, keepdim=True)
    return b


def _body(g, n, spread):
    b = torch.tensor([[0.75], [0.007], [0.007], [0.012]], device="cuda").repeat(1, n)
    if spread:
        b[0] *= _uniform(g, 0.8, 1.2, n)
        b[1:] *= _uniform(g, 0.8, 1.2, 3, n)
    return b.contiguous()


def _states(g, n):
    """float32 [13, n] near hover: positions U[-2, 2]^3, tilt up to 30 degrees, velocities N(0, 0.5^2)."""
    q = _quat(_uniform(g, 0, math.pi / 6, n), torch.randn((3, n), generator=g, device="cuda"))
    return torch.cat((_uniform(g, -2, 2, 3, n), 0.5 * torch.randn((3, n), generator=g, device="cuda"), q,
                      0.2 * torch.randn((3, n), generator=g, device="cuda"))).contiguous()


def _hover(body, split):
    """float32 [8, n] motors at hover."""
    u = torch.zeros((8, body.shape[1]), device="cuda")
    at = 0
    for count, rotors in zip(split, (4, 6, 8)):
        u[:rotors, at:at + count] = body[0, at:at + count] * 9.81 / rotors
        at += count
    return u


def _fleet_inputs(case, seed):
    g, n = _gen(seed), case["n"]
    split = _split(n, case["airframes"])
    body = _body(g, n, case["airframes"] == "mixed")
    md, tg = _commands(g, n, case["modes"], body[0])
    boxes = _boxes(g, case["n_obs"], n) if case["n_obs"] else None
    x0, motors = _states(g, n), _hover(body, split)
    mask = (torch.rand(n, generator=g, device="cuda") < 0.01).to(torch.uint8) if case.get("masked") else None
    return dict(split=split, body=body, modes=md, targets=tg, boxes=boxes, x0=x0, motors=motors, mask=mask)


def _reach_inputs(case, seed):
    g, n = _gen(seed), case["n"]
    split = _split(n, case["airframes"])
    body = _body(g, n, case["airframes"] == "mixed")
    return dict(split=split, body=body, goals=_uniform(g, -1, 1, 3, n), actions=_uniform(g, -0.3, 0.3, n, 4),
                boxes=_boxes(g, case["n_obs"], n) if case["n_obs"] else None)


def _depth_inputs(case, seed):
    g, n = _gen(seed), case["n"]
    boxes, x0 = _boxes(g, case["n_obs"], n), _states(g, n)
    ids = torch.randperm(n, generator=g, device="cuda")[:case["cams"]].to(torch.int32) if case["cams"] < n else None
    return dict(boxes=boxes, x0=x0, ids=ids)


def _adjoint_inputs(case, seed):
    """A fleet near its set points, as gain tuning and command learning have it: no motor reaches its
    limits, where the loss has kinks and the last bit of a state decides a gradient."""
    g, n = _gen(seed), case["n"]
    body = _body(g, n, False)
    q = _quat(_uniform(g, 0, 0.07, n), torch.randn((3, n), generator=g, device="cuda"))
    x0 = torch.cat((_uniform(g, -2, 2, 3, n), 0.1 * torch.randn((3, n), generator=g, device="cuda"), q,
                    0.05 * torch.randn((3, n), generator=g, device="cuda"))).contiguous()
    mix = torch.tensor(MODES[case["modes"]], device="cuda", dtype=torch.uint8)
    md = mix[torch.randint(len(mix), (n,), generator=g, device="cuda")]
    pos = torch.cat((x0[0:3] + _uniform(g, -0.4, 0.4, 3, n), _uniform(g, -0.05, 0.05, 1, n)))
    vel = torch.cat((x0[3:6] + _uniform(g, -0.4, 0.4, 3, n), _uniform(g, -0.2, 0.2, 1, n)))
    att = torch.cat((_uniform(g, -0.1, 0.1, 2, n), _uniform(g, -0.2, 0.2, 1, n), _uniform(g, 0.9, 1.1, 1, n) * (0.75 * 9.81)))
    tg = torch.where(md == 0, pos, torch.where(md == 1, vel, att)).contiguous()
    goal = tg[:3].clone() if case["modes"] == "pos" else x0[0:3] + _uniform(g, -1, 1, 3, n)
    gains = torch.tensor([2, 2, 3, 2, 2, 2, 1.2, 1.2, 0.6, 0.2, 0.2, 0.1]) * (
        1 + 0.1 * torch.rand(12, generator=torch.Generator().manual_seed(int(seed))))
    return dict(body=body, modes=md, targets=tg, x0=x0, motors=_hover(body, (n, 0, 0)), goal=goal, gains=gains,
                weights=_uniform(g, 0.5, 1.5, n))


def _serve_requests(case):
    """(envs, steps, boxes) of each request, ragged."""
    return [(case["n"] * (1 + k % 4) // 2 + 3 * k + 1, case["steps"] * (2 + k % 3) // 3, (8, 0, 32)[k % 3])
            for k in range(case["requests"])]


def _serve_inputs(case, seed):
    g = _gen(seed)
    n = sum(r[0] for r in _serve_requests(case))
    md, tg = _commands(g, n, "all", torch.full((n,), 0.75, device="cuda"))
    return dict(modes=md, targets=tg, boxes=_boxes(g, 32, n))


def _reach_config(case):
    c = _abi.ag_reach_config_default()
    if case["modes"] == "vel":
        c.command_mode = _abi.AG_MODE_BODY_VEL
        c.action_scale[:], c.action_offset[:] = [2, 2, 2, 1], [0, 0, 0, 0]
    return c


# ------------------------------------------------------------- prepare and run --
def prepare(case, seed):
    kind = case["kind"]
    if kind == "reach":
        i = _reach_inputs(case, seed)
        env = ReachEnv(case["n"], goals=i["goals"], task=_reach_config(case), seed=seed, integrator=case["integrator"],
                       substeps_per_step=case["substeps"], n_obstacles=case["n_obs"], n_hexa=i["split"][1],
                       n_octo=i["split"][2])
        env.fleet.set_body(i["body"])
        if case["n_obs"]:
            env.fleet.set_obstacles(i["boxes"])
            env.fleet.set_obstacle_randomization((-5, -5, -5), (5, 5, 5), [
                _abi.box_randomization(euler_min=(-3.1, -1.5, -3.1), euler_max=(3.1, 1.5, 3.1))] * case["n_obs"])
        env.reset()
        return dict(case=case, env=env, actions=i["actions"])
    if kind in ("control", "rollout"):
        i = _fleet_inputs(case, seed)
        fl = Fleet(case["n"], integrator=case["integrator"], substeps_per_step=case["substeps"],
                   n_obstacles=case["n_obs"], n_hexa=i["split"][1], n_octo=i["split"][2], drag=case.get("drag", 0.0),
                   seed=seed)
        fl.set_body(i["body"])
        fl.set_commands(i["modes"], i["targets"])
        if case["n_obs"]:
            fl.set_obstacles(i["boxes"])
        epoch = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
        fl.set_state(i["x0"], i["motors"], epoch)
        fl.synchronize()
        return dict(case=case, fleet=fl, epoch=epoch, seed=seed, **{k: i[k] for k in ("x0", "motors", "targets", "mask")})
    if kind == "depth":
        i = _depth_inputs(case, seed)
        fl = Fleet(case["n"], n_obstacles=case["n_obs"], seed=seed)
        fl.set_obstacles(i["boxes"])
        fl.set_state(i["x0"])
        out = torch.empty((case["cams"], case["height"], case["width"]), device="cuda")
        fl.synchronize()
        return dict(case=case, fleet=fl, ids=i["ids"], out=out)
    if kind == "adjoint":
        i = _adjoint_inputs(case, seed)
        fl = Fleet(case["n"], seed=seed)
        fl.set_commands(i["modes"], i["targets"])
        return dict(case=case, fleet=fl, **i)
    i = _serve_inputs(case, seed)
    pool = RequestPool(i["modes"], i["targets"], i["boxes"].reshape(320, -1))
    requests, at = [], 0
    for k, (n, steps, n_obs) in enumerate(_serve_requests(case)):
        requests.append(pool.request(n_envs=n, n_steps=steps, n_obstacles=n_obs, seed=seed + k, offset=at))
        at += n
    server = Server(max_active=64, hbm_budget_bytes=4 << 30, integrator=case["integrator"],
                    substeps_per_step=case["substeps"])
    return dict(case=case, server=server, pool=pool, requests=requests)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "reach":
        obs, reward, done, info = state["env"].step(state["actions"])
        return dict(obs=obs, reward=reward, done=done, collided=info["collided"])
    if kind == "control":
        fl = state["fleet"]
        fl.set_commands(None, state["targets"])
        fl.step(1)
        return dict(state=fl.state(), epoch=fl.epoch())
    if kind == "rollout":
        fl = state["fleet"]
        fl.set_state(state["x0"], state["motors"], state["epoch"])
        if case["masked"]:
            fl.reset(state["mask"], state["seed"])
        fl.step(case["steps"])
        return dict(state=fl.state(), motors=fl.motors(), epoch=fl.epoch())
    if kind == "depth":
        return state["fleet"].render_depth(case["width"], case["height"], case["hfov"], case["max_range"],
                                           cam_offset=(0.1, -0.02, 0.05) if case["offset"] else None,
                                           env_ids=state["ids"], n_cams=case["cams"], out=state["out"])
    if kind == "adjoint":
        x0, gains = state["x0"].detach().requires_grad_(True), state["gains"].detach().requires_grad_(True)
        targets = state["targets"].detach().requires_grad_(True) if case["targets_grad"] else None
        loss = rollout_loss(state["fleet"], x0, gains, state["motors"], case["steps"], state["goal"], targets=targets)
        loss.backward(state["weights"])
        out = dict(loss=loss.detach(), x0=x0.grad, gains=gains.grad)
        if targets is not None:
            out["targets"] = targets.grad
        return out
    server = state["server"]
    ids = [server.submit(r) for r in state["requests"]]
    return [list(server.wait(i)[:2]) for i in ids]


# -------------------------------------------------------------------- the work --
def _flops_per_substep(integrator):
    """Controller, allocation and integration of one substep (operation counts of the plain equations)."""
    return 883.0 if integrator else 530.0


def work(case):
    kind = case["kind"]
    if kind == "serve":
        sizes = _serve_requests(case)
        steps = sum(n * s for n, s, _ in sizes) * case["substeps"]
        return dict(bytes=float(sum(n * (17 + 56 + 40 * b) for n, _, b in sizes)),
                    flops=steps * _flops_per_substep(case["integrator"]))
    n = case["n"]
    if kind == "depth":
        px = case["cams"] * case["width"] * case["height"]
        return dict(bytes=4.0 * px + case["cams"] * (40.0 * case["n_obs"] + 52), flops=48.0 * px)
    if kind == "adjoint":  # forward 460, reverse 1,217 operations per vehicle-step
        return dict(bytes=n * (52.0 + 16 + 16 + 12 + 52 + 4), flops=1677.0 * n * case["steps"])
    # state, motors, body, mode, targets or action in; state, motors out; boxes in
    rotors = 4.0 if case["airframes"] == "quad" else 5.6
    per_env = 52 + 52 + 8 * rotors + 16 + 1 + 16 + 40 * case["n_obs"]
    if kind == "reach":  # goal, counter in; counter, reward, done, collided, observation out
        per_env += 12 + 4 + 4 + 4 + 1 + 1 + 52
    elif kind == "rollout":  # given states in, states out beside the fleet's own
        per_env += 52 + 4 * rotors + 4
    steps = case.get("steps", 1)
    return dict(bytes=float(per_env * n), flops=n * (steps * case["substeps"] * _flops_per_substep(case["integrator"])
                                                     + 66.0 * case["n_obs"]))


# ----------------------------------------------------------- 64-bit reference --
def _f32(v):
    return float(np.float32(v))


GRAVITY, U_MAX, RADIUS2 = _f32(9.81), 5.0, _f32(_f32(0.2) * _f32(0.2))
DEFAULT_GAINS = [2, 2, 3, 2, 2, 2, _f32(1.2), _f32(1.2), _f32(0.6), _f32(0.2), _f32(0.2), _f32(0.1)]


def _rotors(rotors):
    """Wrench matrix A [4, rotors] and its pseudo-inverse."""
    start = {4: 45.0, 6: 30.0, 8: 22.5}[rotors]
    beta = np.radians(start + 360.0 * np.arange(rotors) / rotors)
    arm, k_yaw = _f32(0.13), _f32(0.016)
    a = np.stack([np.ones(rotors), arm * np.sin(beta), -arm * np.cos(beta), k_yaw * (-1.0) ** np.arange(rotors)])
    to = dict(device="cuda", dtype=torch.float64)
    return torch.tensor(a, **to), torch.tensor(np.linalg.pinv(a), **to)


def _cross(a, b):
    return torch.stack((a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]))


def _dot(a, b):
    return (a * b).sum(0)


def _rotation(q):
    """Columns of R(q), each [3, n], q unit."""
    w, x, y, z = q
    return (torch.stack((1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y))),
            torch.stack((2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x))),
            torch.stack((2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y))))


def _quat_rate(q, w):
    return 0.5 * torch.stack((-q[1] * w[0] - q[2] * w[1] - q[3] * w[2], q[0] * w[0] + q[2] * w[2] - q[3] * w[1],
                              q[0] * w[1] + q[3] * w[0] - q[1] * w[2], q[0] * w[2] + q[1] * w[1] - q[2] * w[0]))


def _controller(s, md, present, tg, body, gains):
    """Commanded (f, M) [4, n] of the geometric controller; s = (p, v, q, w)."""
    p, v, q, w = s
    m, inertia = body[0], body[1:]
    kx, kv, kr, kw = (gains[3 * i:3 * i + 3, None] for i in range(4))
    cols = _rotation(q)
    b3, zero, one = cols[2], torch.zeros_like(m), torch.ones_like(m)
    e3 = torch.stack((zero, zero, one))
    f = rate = rd = None

    def choose(new, old, mode):
        return new if old is None else torch.where(md == mode, new, old)

    for mode in present:
        if mode == 0:
            a = -kx * (p - tg[:3]) - kv * v + GRAVITY * e3
            d3 = a / a.norm(dim=0, keepdim=True)
            d2 = _cross(d3, torch.stack((torch.cos(tg[3]), torch.sin(tg[3]), zero)))
            d2 = d2 / d2.norm(dim=0, keepdim=True)
            fm, rm, dm = m * _dot(a, b3), zero, (_cross(d2, d3), d2, d3)
        else:
            psi = torch.atan2(cols[0][1], cols[0][0])
            cp, sp = torch.cos(psi), torch.sin(psi)
            if mode == 1:
                vv = torch.stack((cp * v[0] + sp * v[1], -sp * v[0] + cp * v[1], v[2]))
                a = kv * (tg[:3] - vv) + GRAVITY * e3
                fm = m * _dot(a, torch.stack((cp * b3[0] + sp * b3[1], -sp * b3[0] + cp * b3[1], b3[2])))
                phi, theta = torch.atan2(-a[1], torch.sqrt(a[0] ** 2 + a[2] ** 2)), torch.atan2(a[0], a[2])
                rm = tg[3]
            else:
                phi, theta, rm, fm = tg[0], tg[1], tg[2], tg[3]
            cf, sf, ct, st = torch.cos(phi), torch.sin(phi), torch.cos(theta), torch.sin(theta)
            dm = tuple(torch.stack((cp * x - sp * y, sp * x + cp * y, z)) for x, y, z in (
                (ct, zero, -st), (st * sf, cf, ct * sf), (st * cf, -sf, ct * cf)))
        rd = dm if rd is None else tuple(choose(x, y, mode) for x, y in zip(dm, rd))
        f, rate = choose(fm, f, mode), choose(rm, rate, mode)
    er = 0.5 * torch.stack((_dot(rd[2], cols[1]) - _dot(rd[1], cols[2]), _dot(rd[0], cols[2]) - _dot(rd[2], cols[0]),
                            _dot(rd[1], cols[0]) - _dot(rd[0], cols[1])))
    ew = w - rate * torch.stack((cols[0][2], cols[1][2], cols[2][2]))
    return torch.cat((f[None], -kr * er - kw * ew + _cross(w, inertia * w))), b3


def _substep(s, u, md, present, tg, body, gains, rotors, h, alpha, drag, integrator):
    cmd, b3 = _controller(s, md, present, tg, body, gains)
    a, pinv = rotors
    u = u + alpha * (torch.clamp(pinv @ cmd, 0, U_MAX) - u)
    wrench = a @ u
    p, v, q, w = s
    m, inertia = body[0], body[1:]
    down = torch.tensor([[0.0], [0.0], [-GRAVITY]], device="cuda", dtype=torch.float64)

    def linear(axis, v):
        return wrench[0] / m * axis - (drag / m) * v + down

    def angular(w):
        return (wrench[1:] - _cross(w, inertia * w)) / inertia

    if not integrator:
        v2, w2 = v + h * linear(b3, v), w + h * angular(w)
        p2, q2 = p + h * v2, q + h * _quat_rate(q, w2)
    else:
        def rates(v, q, w):
            return v, linear(_rotation(q / q.norm(dim=0, keepdim=True))[2], v), _quat_rate(q, w), angular(w)

        k = rates(v, q, w)
        total = list(k)
        for c, weight in ((0.5 * h, 2), (0.5 * h, 2), (h, 1)):
            k = rates(v + c * k[1], q + c * k[2], w + c * k[3])
            total = [t + weight * x for t, x in zip(total, k)]
        p2, v2, q2, w2 = (x + h / 6 * t for x, t in zip(s, total))
    return (p2, v2, q2 / q2.norm(dim=0, keepdim=True), w2), u


def _philox(c, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(a, x):
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        return (hi + (lo >> 16)) >> 16, (((hi & 0xFFFF) << 16) + lo) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _reset_draw(env, epoch, seed):
    """States (p, v, q, w) of the reset draw; env, epoch, seed int64 [n]."""
    unit = [[(w >> 8).double() / 2.0 ** 24 for w in _philox((env, epoch, torch.full_like(env, slot), torch.zeros_like(env)),
                                                            seed & 0xFFFFFFFF, seed >> 32)] for slot in range(3)]
    p = torch.stack([-2 + 4 * x for x in unit[0][:3]])
    az, turn, half = 1 - 2 * unit[0][3], 2 * math.pi * unit[1][0], _f32(math.pi / 12) * unit[1][1]
    rho = torch.sqrt(torch.clamp(1 - az * az, min=0))
    q = torch.stack((torch.cos(half), torch.sin(half) * rho * torch.cos(turn), torch.sin(half) * rho * torch.sin(turn),
                     torch.sin(half) * az))
    r1, r2 = (torch.sqrt(-2 * torch.log(x + 2.0 ** -24)) for x in (unit[1][2], unit[2][0]))
    t1, t2 = 2 * math.pi * unit[1][3], 2 * math.pi * unit[2][1]
    return p, 0.5 * torch.stack((r1 * torch.cos(t1), r1 * torch.sin(t1), r2 * torch.cos(t2))), q, torch.zeros_like(p)


def _hits(p, boxes):
    """Whether the vehicle sphere touches a box; boxes [n_obs, 10, n]."""
    d = p[None] - boxes[:, 0:3]
    w, u = boxes[:, 6:7], boxes[:, 7:10]
    t = 2 * torch.cross(u, d, dim=1)
    local = d - w * t + torch.cross(u, t, dim=1)
    e = torch.clamp(local.abs() - boxes[:, 3:6], min=0)
    return ((e * e).sum(1) <= RADIUS2).any(0)


def _pick(mask, new, old):
    return tuple(torch.where(mask, x, y) for x, y in zip(new, old))


def _simulate(s, u, md, modes, tg, body, n_rotors, boxes, env, seed, epoch, case, steps, horizon=None):
    """`steps` steps of one airframe with collision resets; horizon [n]: steps of each environment.
    Returns the state, the motors and who collided in the last step."""
    substeps, drag = case["substeps"], _f32(case.get("drag", 0.0))
    h = _f32(0.01) / substeps
    alpha = 1 - math.exp(-h / _f32(0.03))
    rotors = _rotors(n_rotors)
    gains = torch.tensor(DEFAULT_GAINS, device="cuda", dtype=torch.float64)
    hit = torch.zeros_like(body[0], dtype=torch.bool)
    for step in range(steps):
        s2, u2 = s, u
        for _ in range(substeps):
            s2, u2 = _substep(s2, u2, md, modes, tg, body, gains, rotors, h, alpha, drag, case["integrator"])
        if boxes is not None:
            hit = _hits(s2[0], boxes)
            if horizon is not None:
                hit = hit & (step < horizon)
            if bool(hit.any()):
                epoch = epoch + hit
                s2 = _pick(hit, _reset_draw(env, epoch, seed), s2)
                u2 = torch.where(hit, (body[0] * GRAVITY / n_rotors).expand_as(u2), u2)
        if horizon is not None:
            live = step < horizon
            s2, u2 = _pick(live, s2, s), torch.where(live, u2, u)
        s, u = s2, u2
    return s, u, hit


def _by_airframe(split, run_range):
    """run_range(lo, hi, rotors) over each airframe's range; results joined along the environments."""
    parts, at = [], 0
    for count, rotors in zip(split, (4, 6, 8)):
        if count:
            parts.append(run_range(at, at + count, rotors))
        at += count
    return [torch.cat(x, dim=-1) for x in zip(*parts)]


def _seconds(n, substeps, integrator):
    """About how long the 64-bit simulation takes."""
    return substeps * (700 if integrator else 300) * max(9e-6, n * 3 * 24 / 4e12)


def _exact_fleet(case, seed):
    steps = case.get("steps", 1)
    if _seconds(case["n"], steps * case["substeps"], case["integrator"]) > 12:
        return None
    i = _fleet_inputs(case, seed)

    def one(lo, hi, n_rotors):
        env = torch.arange(lo, hi, device="cuda")
        body, x0 = i["body"][:, lo:hi].double(), i["x0"][:, lo:hi].double()
        u = i["motors"][:n_rotors, lo:hi].double()
        s = (x0[0:3], x0[3:6], x0[6:10] / x0[6:10].norm(dim=0, keepdim=True), x0[10:13])
        epoch, key = torch.zeros_like(env), torch.full_like(env, seed)
        if case.get("masked"):
            mask = i["mask"][lo:hi] != 0
            epoch = epoch + mask
            s = _pick(mask, _reset_draw(env, epoch, key), s)
            u = torch.where(mask, (body[0] * GRAVITY / n_rotors).expand_as(u), u)
        boxes = None if i["boxes"] is None else i["boxes"][:, :, lo:hi].double()
        s, u, _ = _simulate(s, u, i["modes"][lo:hi], MODES[case["modes"]], i["targets"][:, lo:hi].double(), body, n_rotors,
                            boxes, env, key, epoch, case, steps)
        return torch.cat(s), torch.cat((u, torch.zeros((8 - n_rotors, hi - lo), device="cuda", dtype=torch.float64)))

    state, motors = _by_airframe(i["split"], one)
    if case["kind"] == "control":
        return dict(state=state, epoch=None)
    return dict(state=state, motors=motors, epoch=None)


def _exact_reach(case, seed):
    i, mode = _reach_inputs(case, seed), MODES[case["modes"]]
    if case["modes"] == "vel":
        scale, offset = [2, 2, 2, 1], [0, 0, 0, 0]
    else:
        mg = np.float32(0.75) * np.float32(9.81)
        scale = [_f32(0.52359878), _f32(0.52359878), 1.0, float(np.float32(0.5) * mg)]
        offset = [0, 0, 0, float(mg)]
    scale, offset = (torch.tensor(x, device="cuda", dtype=torch.float64)[:, None] for x in (scale, offset))
    tg_all, goals = offset + scale * i["actions"].double().t().clamp(-1, 1), i["goals"].double()

    def one(lo, hi, n_rotors):
        env = torch.arange(lo, hi, device="cuda")
        key, first = torch.full_like(env, seed), torch.ones_like(env)
        body, goal = i["body"][:, lo:hi].double(), goals[:, lo:hi]
        u = (body[0] * GRAVITY / n_rotors).expand(n_rotors, -1)
        boxes = None
        if case["n_obs"]:  # the first reset re-placed every box: see ag_set_obstacle_randomization
            boxes = _replaced(i["boxes"][:, :, lo:hi].double(), env, first, key)
        md = torch.full_like(env, mode[0], dtype=torch.uint8)
        still = dict(case, steps=1)
        start = _reset_draw(env, first, key)
        s = (start[0], start[1], start[2] / start[2].norm(dim=0, keepdim=True), start[3])
        s, _, hit = _simulate(s, u, md, mode, tg_all[:, lo:hi], body, n_rotors, boxes, env, key, first, still, 1)
        dist = (s[0] - goal).norm(dim=0)
        reward = torch.where(hit, torch.full_like(dist, -10.0), -(dist + _f32(0.1) * s[1].norm(dim=0) +
                                                                  _f32(0.01) * s[3].norm(dim=0)))
        s = _pick(~hit & (dist > 8.0), _reset_draw(env, first + 1, key), s)
        sign = torch.where(s[2][0] < 0, -1.0, 1.0)
        return torch.cat((s[0] - goal, s[1], sign * s[2], s[3])), reward

    obs, reward = _by_airframe(i["split"], one)
    return dict(obs=obs.t().contiguous(), reward=reward, done=None, collided=None)


def _replaced(boxes, env, epoch, seed):
    """Every box at its re-drawn pose: centres U[-5, 5]^3, roll, pitch, yaw within +-(3.1, 1.5, 3.1)."""
    out = boxes.clone()
    lo, hi = [-_f32(3.1), -_f32(1.5), -_f32(3.1)], [_f32(3.1), _f32(1.5), _f32(3.1)]
    for k in range(len(boxes)):
        unit = [[(w >> 8).double() / 2.0 ** 24 for w in _philox(
            (env, epoch, torch.full_like(env, k), torch.full_like(env, slot)), seed & 0xFFFFFFFF, seed >> 32)]
            for slot in (1, 2)]
        out[k, 0:3] = torch.stack([-5 + 10 * x for x in unit[0][:3]])
        half = [0.5 * (a + (b - a) * x) for a, b, x in zip(lo, hi, (unit[0][3], unit[1][0], unit[1][1]))]
        (cr, cp, cy), (sr, sp, sy) = [torch.cos(x) for x in half], [torch.sin(x) for x in half]
        out[k, 6:10] = torch.stack((cy * cp * cr + sy * sp * sr, cy * cp * sr - sy * sp * cr,
                                    cy * sp * cr + sy * cp * sr, sy * cp * cr - cy * sp * sr))
    return out


def _exact_depth(case, seed):
    i = _depth_inputs(case, seed)
    ids = torch.arange(case["cams"], device="cuda") if i["ids"] is None else i["ids"].long()
    width, height = case["width"], case["height"]
    to = dict(device="cuda", dtype=torch.float64)
    inv_f = math.tan(0.5 * _f32(case["hfov"])) / (0.5 * width)
    dy = (-(torch.arange(width, **to) + 0.5 - 0.5 * width) * inv_f)[None, None, :]
    dz = (-(torch.arange(height, **to) + 0.5 - 0.5 * height) * inv_f)[None, :, None]
    mount = torch.tensor([_f32(0.1), _f32(-0.02), _f32(0.05)] if case["offset"] else [0.0, 0.0, 0.0], **to)
    images, most = [], max(1, (1 << 23) // (width * height))
    for at in range(0, len(ids), most):
        env = ids[at:at + most]
        x0 = i["x0"][:, env].double()
        cam = torch.stack(_rotation(x0[6:10] / x0[6:10].norm(dim=0, keepdim=True)), dim=1)  # [3, 3, c]: R[i][j]
        origin = x0[0:3] + (cam * mount[None, :, None]).sum(1)
        best = torch.full((len(env), height, width), _f32(case["max_range"]), **to)
        for k in range(case["n_obs"]):
            b = i["boxes"][k][:, env].double()
            box = torch.stack(_rotation(b[6:10]), dim=1)
            m = torch.einsum("aic,ajc->cij", box, cam)  # the camera's axes in the box frame
            o = torch.einsum("aic,ac->ic", box, origin - b[0:3])
            near, far = torch.zeros_like(best), torch.full_like(best, math.inf)
            for ax in range(3):
                d = m[:, ax, 0, None, None] + m[:, ax, 1, None, None] * dy + m[:, ax, 2, None, None] * dz
                t0, t1 = ((sgn * b[3 + ax] - o[ax])[:, None, None] / d for sgn in (-1, 1))
                near, far = torch.maximum(near, torch.minimum(t0, t1)), torch.minimum(far, torch.maximum(t0, t1))
            best = torch.where(near <= torch.minimum(far, best), near, best)
        images.append(best)
    return torch.cat(images)


def _exact_adjoint(case, seed):
    i, steps = _adjoint_inputs(case, seed), case["steps"]
    if _seconds(case["n"], 5 * steps, 0) > 15:
        return None
    body, modes, md = i["body"].double(), MODES[case["modes"]], i["modes"]
    h = _f32(0.01)
    alpha = 1 - math.exp(-h / _f32(0.03))
    rotors = _rotors(4)
    x0 = i["x0"].double().requires_grad_(True)
    gains_in = i["gains"].double().requires_grad_(True)
    tg = i["targets"].double().requires_grad_(bool(case["targets_grad"]))
    goal, w_omega = i["goal"].double(), _f32(0.01)

    def segment(count, p, v, q, w, u, gains, tg, total):
        s = (p, v, q, w)
        for _ in range(count):
            s, u = _substep(s, u, md, modes, tg, body, gains, rotors, h, alpha, 0.0, 0)
            e = s[0] - goal
            total = total + _dot(e, e) + w_omega * _dot(s[3], s[3])
        return (*s, u, total)

    with torch.enable_grad():
        gains = gains_in.cuda()
        s = (x0[0:3], x0[3:6], x0[6:10] / x0[6:10].norm(dim=0, keepdim=True), x0[10:13], i["motors"][:4].double())
        total = torch.zeros_like(body[0])
        for at in range(0, steps, 16):
            *s, total = checkpoint(segment, min(16, steps - at), *s, gains, tg, total, use_reentrant=False)
        total.backward(i["weights"].double())
    out = dict(loss=total.detach(), x0=x0.grad, gains=gains_in.grad)
    if case["targets_grad"]:
        out["targets"] = tg.grad
    return out


def _exact_serve(case, seed):
    sizes = _serve_requests(case)
    n, steps = sum(r[0] for r in sizes), max(r[1] for r in sizes)
    if _seconds(n, steps * case["substeps"], case["integrator"]) > 12:
        return None
    i = _serve_inputs(case, seed)
    to = dict(device="cuda")
    env = torch.cat([torch.arange(r[0], **to) for r in sizes])
    key = torch.cat([torch.full((r[0],), seed + k, **to) for k, r in enumerate(sizes)])
    horizon = torch.cat([torch.full((r[0],), r[1], **to) for r in sizes])
    boxes = i["boxes"].double()
    used = torch.cat([torch.full((r[0],), r[2], **to) for r in sizes])
    boxes[:, 0] = torch.where(torch.arange(32, **to)[:, None] < used, boxes[:, 0], 1e9)  # boxes beyond a request's own
    body = _body(None, n, False).double()
    epoch = torch.ones_like(env)
    p, v, q, w = _reset_draw(env, epoch, key)
    u = (body[0] * GRAVITY / 4).expand(4, -1)
    s, _, _ = _simulate((p, v, q / q.norm(dim=0, keepdim=True), w), u, i["modes"], MODES["all"], i["targets"].double(),
                        body, 4, boxes, env, key, epoch, case, steps, horizon)
    state, out, at = torch.cat(s), [], 0
    for r in sizes:
        out.append([state[:, at:at + r[0]].cpu().numpy(), None])
        at += r[0]
    return out


def exact(case, seed):
    with torch.no_grad():
        return {"reach": _exact_reach, "control": _exact_fleet, "rollout": _exact_fleet, "depth": _exact_depth,
                "adjoint": _exact_adjoint, "serve": _exact_serve}[case["kind"]](case, seed)
