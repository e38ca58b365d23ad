"""The grouping order pads each (rotor type, command mode) run to whole warps:
at sizes around its window and warp edges every environment is stepped exactly
once, by the loop of its own mode, and recorded and swept once by the adjoint."""
import numpy as np
import pytest
import torch

from paper_2305_16510_gb300 import _abi, workloads as W

from harness import gpu_fleet

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 32, 33, 1023, 1025, 16383, 16384, 16385, 2 * 16384 + 1000]


def _workload(n, mixed):
    hexa, octo = (n // 3, n // 4) if mixed else (0, 0)
    return W.Workload("order", n, 1, 0, 0, n - hexa - octo, hexa, octo, drag=0.1, mass_rand=0.2, mode_mix=(0, 1, 2, 3))


@pytest.mark.parametrize("mixed", [False, True], ids=["quads", "mixed"])
@pytest.mark.parametrize("n", SIZES)
def test_grouped_order_steps_every_environment_once(n, mixed, monkeypatch):
    w = _workload(n, mixed)
    inp = W.make_inputs(w, 3)
    outs = []
    for order in ("grouped", "identity"):
        monkeypatch.setenv("AG_FUSED_ORDER", order)
        fl = gpu_fleet(w, inp, 3)
        fl.reset(None, 3)
        fl.step(5)
        outs.append((fl.state().cpu().numpy(), fl.motors().cpu().numpy(), fl.epoch().cpu().numpy()))
        fl.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    assert (outs[0][2] == 1).all()


@pytest.mark.parametrize("n", SIZES)
def test_adjoint_does_not_depend_on_a_vehicles_slot(n):
    """The same quads in the opposite order: each one's loss and gradients are the same bits."""
    w = _workload(n, False)
    inp = W.make_inputs(w, 4)
    outs = []
    for flip in (False, True):
        turn = (lambda a: a[..., ::-1].copy()) if flip else (lambda a: a)
        fl = gpu_fleet(w, W.Inputs(turn(inp.modes), turn(inp.targets), turn(inp.body), None), 4)
        st = np.random.default_rng(6).uniform(-1, 1, (13, n)).astype(np.float32)
        st[6] = 2.0
        fl.set_state(turn(st), turn(np.full((8, n), 1.8, np.float32)))
        loss, gx, gge, gt = (torch.empty(s, device="cuda") for s in ((n,), (13, n), (12, n), (4, n)))
        _abi.ag_rollout_loss(fl.ctx, 9, 1.0, 0.1, torch.zeros((3, n), device="cuda"), loss)
        _abi.ag_backward(fl.ctx, None, gx, None, gge, gt)
        outs.append([turn(t.cpu().numpy()) for t in (loss, gx, gge, gt)] + [turn(fl.state().cpu().numpy())])
        fl.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    assert np.isfinite(outs[0][1]).all() and (np.abs(outs[0][1]).sum(axis=0) > 0).all()


@pytest.mark.parametrize("n", [1024, 3000, 4095, 4096, 4097, 9000, 16384 + 4097])
def test_order_around_the_sizes_of_its_kernels(n, monkeypatch):
    """Fleets of up to 1,024 and 4,096 environments are ordered in fewer rounds."""
    w = _workload(n, True)
    inp = W.make_inputs(w, 3)
    outs = []
    for order in ("grouped", "identity"):
        monkeypatch.setenv("AG_FUSED_ORDER", order)
        fl = gpu_fleet(w, inp, 3)
        fl.set_commands(modes=inp.modes[::-1].copy())   # another order over the first one
        fl.reset(None, 3)
        fl.step(3)
        outs.append((fl.state().cpu().numpy(), fl.motors().cpu().numpy()))
        fl.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
