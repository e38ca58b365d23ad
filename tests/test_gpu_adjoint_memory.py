"""The recorded rollout and its gradient by where their arguments lie: arrays
in aligned memory of the context's device are read and written in place, any
other, and those that overlap, through the context's own buffers. The results
are the same bits, with the whole-horizon tape and with the one-segment tape.
A change of command modes after the record leaves the recording as it is."""
import numpy as np
import pytest
import torch

from paper_2305_16510_gb300 import _abi, workloads as W
from paper_2305_16510_gb300.fleet import Fleet

pytestmark = pytest.mark.gpu
H, SEED = 40, 8
BUDGET = {"whole": 0, "segment": 200_000}  # the second is too small for the whole horizon


def _inputs(n):
    w = W.Workload("adjoint memory", n, 1, 0, 0, n, 0, 0, mode_mix=(0, 1, 2, 3))
    return W.make_inputs(w, SEED), np.random.default_rng(SEED)


def _fleet(inp, n, tape):
    fl = Fleet(n, motor_tau=0.03, seed=SEED, hbm_budget_bytes=BUDGET[tape])
    fl.set_body(inp.body)
    fl.set_commands(inp.modes, inp.targets)
    fl.reset(None, SEED)
    return fl


class _Place:
    """Arrays in one kind of memory: addresses to pass, values read back later."""

    def __init__(self, kind):
        self.kind = kind

    def put(self, a):
        a = np.ascontiguousarray(a, np.float32)
        if self.kind == "host":
            return a.copy()
        if self.kind == "pinned":
            return torch.from_numpy(a.copy()).pin_memory()
        if self.kind == "device":
            return torch.from_numpy(a).cuda()
        raw = torch.zeros(a.nbytes + 4, dtype=torch.uint8, device="cuda")  # device memory at an odd address
        raw[2:2 + a.nbytes] = torch.from_numpy(a.view(np.uint8).reshape(-1)).cuda()
        return raw

    def arg(self, x):
        return x if self.kind != "odd" else x.data_ptr() + 2

    def get(self, x, shape):
        if self.kind == "host":
            return x.reshape(shape)
        if self.kind == "odd":
            count = int(np.prod(shape))
            return x[2:2 + 4 * count].cpu().numpy().copy().view(np.float32).reshape(shape)
        return x.cpu().numpy().reshape(shape)


def _gradients(fl, n, goal, weights, place, outs=("gx", "gg", "gge", "gt")):
    """Loss and the wanted gradients with every argument in `place`."""
    shapes = {"gx": (13, n), "gg": (12,), "gge": (12, n), "gt": (4, n)}
    g, w, loss = place.put(goal), place.put(weights), place.put(np.zeros(n))
    out = {k: place.put(np.full(s, 7.0)) for k, s in shapes.items() if k in outs}
    _abi.ag_rollout_loss(fl.ctx, H, 1.0, 0.1, place.arg(g), place.arg(loss))
    args = [place.arg(out[k]) if k in out else None for k in ("gx", "gg", "gge", "gt")]
    _abi.ag_backward(fl.ctx, place.arg(w), *args)
    fl.synchronize()
    return {"loss": place.get(loss, (n,)), **{k: place.get(v, shapes[k]) for k, v in out.items()}}


@pytest.mark.parametrize("tape", ["whole", "segment"])
def test_results_do_not_depend_on_where_arguments_lie(tape):
    n = 300
    inp, rng = _inputs(n)
    goal, weights = rng.uniform(-1, 1, (3, n)), rng.uniform(0.5, 1.5, n)
    got = {}
    for kind in ("device", "host", "pinned", "odd"):
        fl = _fleet(inp, n, tape)
        got[kind] = _gradients(fl, n, goal, weights, _Place(kind))
        fl.close()
    assert np.isfinite(got["device"]["gx"]).all() and np.abs(got["device"]["gg"]).min() > 0
    for kind in ("host", "pinned", "odd"):
        for k, v in got["device"].items():
            np.testing.assert_array_equal(got[kind][k], v, err_msg=f"{kind} {k}")
    for outs in (("gx",), ("gg", "gt"), ("gge",)):   # some outputs only, host and device mixed over the calls
        for kind in ("device", "host"):
            fl = _fleet(inp, n, tape)
            part = _gradients(fl, n, goal, weights, _Place(kind), outs)
            fl.close()
            for k, v in part.items():
                np.testing.assert_array_equal(v, got["device"][k], err_msg=f"{outs} {kind} {k}")


@pytest.mark.parametrize("tape", ["whole", "segment"])
def test_overlapping_arguments(tape):
    """The loss over the goals' second row, the loss weights in the middle of an output."""
    n = 300
    inp, rng = _inputs(n)
    goal, weights = rng.uniform(-1, 1, (3, n)), rng.uniform(0.5, 1.5, n)
    fl = _fleet(inp, n, tape)
    want = _gradients(fl, n, goal, weights, _Place("device"))
    fl.close()
    for target in ("gx", "gt"):
        fl = _fleet(inp, n, tape)
        g = torch.from_numpy(goal.astype(np.float32)).cuda()
        _abi.ag_rollout_loss(fl.ctx, H, 1.0, 0.1, g, g[1])
        gx, gt = torch.zeros((13, n), device="cuda"), torch.zeros((4, n), device="cuda")
        w = (gx if target == "gx" else gt)[2]
        w.copy_(torch.from_numpy(weights.astype(np.float32)))
        _abi.ag_backward(fl.ctx, w, gx, None, None, gt)
        fl.synchronize()
        np.testing.assert_array_equal(g[1].cpu().numpy(), want["loss"])
        np.testing.assert_array_equal(gx.cpu().numpy(), want["gx"])
        np.testing.assert_array_equal(gt.cpu().numpy(), want["gt"])
        fl.close()


@pytest.mark.parametrize("how", ["commands", "task"])
@pytest.mark.parametrize("tape", ["whole", "segment"])
def test_recording_survives_a_change_of_modes(tape, how):
    """Other modes regroup the thread slots: a backward after that is still the recorded rollout's."""
    n = 300
    inp, rng = _inputs(n)
    goal = torch.from_numpy(rng.uniform(-1, 1, (3, n)).astype(np.float32)).cuda()
    outs = []
    for change in (False, True):
        fl = _fleet(inp, n, tape)
        loss = torch.empty(n, device="cuda")
        _abi.ag_rollout_loss(fl.ctx, H, 1.0, 0.1, goal, loss)
        for _ in range(2 if change else 0):   # the second change finds the recording already set aside
            if how == "commands":
                fl.set_commands(modes=rng.integers(0, 4, n).astype(np.uint8))
            else:
                _abi.ag_reach_begin(fl.ctx, _abi.ag_reach_config_default(), goal)
        gx, gge, gt = (torch.empty((r, n), device="cuda") for r in (13, 12, 4))
        _abi.ag_backward(fl.ctx, None, gx, None, gge, gt)
        outs.append([t.cpu().numpy() for t in (gx, gge, gt)])
        fl.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)


def test_checkpoints_of_a_small_fleet_take_no_padding():
    """One quad, a checkpoint every step for 40,000 steps: 3.4 MB (the order's padding would make it 323 MB)."""
    n, steps = 1, 40_000
    c = _abi.ag_config_default()
    c.n_envs = c.n_quad = n
    c.record_every, c.hbm_budget_bytes = 1, 100_000
    ctx = _abi.ag_create(c, torch.cuda.current_stream().cuda_stream)
    goal, loss = torch.zeros((3, n), device="cuda"), torch.empty(n, device="cuda")
    gx = torch.empty((13, n), device="cuda")
    _abi.ag_rollout_loss(ctx, 1, 1.0, 0.1, goal, loss)    # the buffers that do not grow with the horizon
    _abi.ag_synchronize(ctx)
    free, _ = torch.cuda.mem_get_info()
    _abi.ag_rollout_loss(ctx, steps, 1.0, 0.1, goal, loss)
    _abi.ag_synchronize(ctx)
    assert free - torch.cuda.mem_get_info()[0] < 32 << 20
    _abi.ag_backward(ctx, None, gx, None, None, None)
    _abi.ag_synchronize(ctx)
    assert torch.isfinite(loss).all()
    _abi.ag_destroy(ctx)
