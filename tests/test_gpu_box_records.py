"""Box records: the collision test reads every box's circumscribed sphere and
runs the exact sphere-vs-box test only on those within reach. Its decisions
must be those of the exact test on every box (AG_FUSED_SKIP=0), bit for bit,
and the records must hold what ag_set_obstacles was given."""
import numpy as np
import pytest
import torch

from paper_2305_16510_gb300 import workloads as W
from paper_2305_16510_gb300.fleet import Fleet
from paper_2305_16510_gb300.task import ReachEnv

from harness import box_margin, gpu_fleet

pytestmark = pytest.mark.gpu


def _case(n_obs, seed):
    """Long thin, flat and large boxes around the vehicles, quaternion norms off
    by up to the admitted 1e-4 of the squared norm, some vehicles at positions
    that are huge or not finite."""
    n = 3001
    w = W.Workload("records", n, 2, 1, n_obs, n, 0, 0, mode_mix=(0, 1, 2, 3))
    inp = W.make_inputs(w, seed)
    rng = np.random.default_rng(seed)
    boxes = inp.boxes.copy()
    boxes[:, 0:3] = rng.uniform(-3, 3, (n_obs, 3, n))
    boxes[:, 3:6] = rng.choice([0.01, 0.1, 0.5, 2.5], (n_obs, 3, n)) / np.sqrt(n_obs)
    boxes[:, 6:10] *= np.sqrt(1 + rng.uniform(-9e-5, 9e-5, (n_obs, 1, n)))
    return w, W.Inputs(inp.modes, inp.targets, inp.body, np.ascontiguousarray(boxes, np.float32))


@pytest.mark.parametrize("n_obs", [1, 2, 31, 32, 33, 64])
def test_sphere_first_tests_decide_as_the_exact_test(n_obs, monkeypatch):
    w, inp = _case(n_obs, 60 + n_obs)
    outs = []
    for skip in ("1", "0"):
        monkeypatch.setenv("AG_FUSED_SKIP", skip)
        fl = gpu_fleet(w, inp, 5)
        fl.reset(None, 5)
        st = fl.state()
        st[0:3, 0:40:8] = torch.tensor([float("inf"), float("nan"), -float("inf"), 1e19, 3e38], device="cuda")
        st[0, 3:43:8] = 1e20
        st[1, 4:44:8] = -2e6
        fl.set_state(st)
        got = []
        for steps in (1, 1, 1, 7, 60):   # single steps want only the decision, longer calls the clearance too
            fl.step(steps)
            col, ids = fl.events()
            got += [fl.state(), fl.motors(), fl.epoch(), col, ids.sort().values]
        outs.append([t.cpu().numpy() for t in got])
        fl.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    assert (outs[0][-3] > 1).sum() > 50   # collisions happened


@pytest.mark.parametrize("n_obs", [1, 3])
def test_obstacles_round_trip_from_host_and_device(n_obs):
    w, inp = _case(n_obs, 7)
    fl = gpu_fleet(w, inp, 5)
    np.testing.assert_array_equal(fl.obstacles().cpu().numpy(), inp.boxes)
    from paper_2305_16510_gb300 import _abi
    _abi.ag_set_obstacles(fl.ctx, inp.boxes[:, :, ::-1].copy())        # pageable host memory
    host = np.empty_like(inp.boxes)
    _abi.ag_get_obstacles(fl.ctx, host)
    fl.synchronize()
    np.testing.assert_array_equal(host, inp.boxes[:, :, ::-1])
    fl.close()


@pytest.mark.parametrize("steps", [1, 3])
@pytest.mark.parametrize("n_obs", [1, 9])
def test_vehicle_at_a_box_centre_collides(n_obs, steps, monkeypatch):
    """Vehicles from 1e-24 to 1e-16 m off a box's centre, where the squared
    distance is zero, subnormal or the smallest normal numbers: every one is
    inside the box, in the fused step and in the task step."""
    offs = np.concatenate([[0.0], np.geomspace(1e-24, 1e-16, 200)]).astype(np.float32)
    dirs = np.array([[1, 0, 0], [0, -1, 0], [0, 0, 1], [1, 1, 1]], np.float32)
    p = (dirs[:, :, None] * offs).transpose(1, 0, 2).reshape(3, -1)
    n = p.shape[1]
    boxes = np.zeros((n_obs, 10, n), np.float32)
    boxes[:, 3:6], boxes[:, 6] = 0.1, 1.0
    boxes[1:, 0] = 30.0                    # only the first box is near
    st = np.zeros((13, n), np.float32)
    st[0:3], st[6] = p, 1.0
    for skip in ("1", "0"):
        monkeypatch.setenv("AG_FUSED_SKIP", skip)
        fl = Fleet(n, n_obstacles=n_obs, dt=1e-30, seed=4)   # so short a step that nothing moves
        fl.set_obstacles(boxes)
        fl.set_state(st)
        fl.step(steps)
        col, ids = fl.events()
        assert bool(col.all()) and ids.numel() == n
        fl.close()
    env = ReachEnv(n, n_obstacles=n_obs, dt=1e-30, seed=4)
    env.fleet.set_obstacles(boxes)
    env.reset()
    env.fleet.set_state(st)
    *_, info = env.step(torch.zeros((n, 4), device="cuda"))
    assert bool(info["collided"].all())
    env.close()


@pytest.mark.parametrize("n,n_obs,budget", [(1001, 5, 0), (700_001, 10, 0), (1000, 5, 516_000), (1000, 5, 475_000)])
def test_obstacles_from_host_memory_in_several_parts(n, n_obs, budget):
    """All boxes at once; nine and then one (more rows than 256 MB); two and one
    at a time, which is what the budgets leave."""
    from paper_2305_16510_gb300 import _abi
    rng = np.random.default_rng(n)
    boxes = rng.uniform(0.1, 5.0, (n_obs, 10, n)).astype(np.float32)
    boxes[:, 6:10] = 0.5
    fl = Fleet(n, n_obstacles=n_obs, hbm_budget_bytes=budget)
    for memory in (boxes, torch.from_numpy(boxes).pin_memory()):
        fl.set_obstacles(np.full((n_obs, 10, n), 0.5, np.float32))
        _abi.ag_set_obstacles(fl.ctx, memory)
        np.testing.assert_array_equal(fl.obstacles().cpu().numpy(), boxes)
        host = np.zeros_like(boxes)
        _abi.ag_get_obstacles(fl.ctx, host)
        fl.synchronize()
        np.testing.assert_array_equal(host, boxes)
    fl.close()


@pytest.mark.parametrize("steps", [1, 2])
@pytest.mark.parametrize("n_obs", [1, 2, 3, 4, 5, 7, 33, 64])
def test_decisions_among_walls_and_small_boxes(n_obs, steps):
    """Calls of one step have a kernel of their own, which tests marked boxes four
    at a time. Walls, whose spheres mark every box, and small boxes: with so
    short a step that nothing moves, the flags are those of the float64 distances,
    but for near ties (the squared distances are good to 1e-5 m^2)."""
    n = 4000
    rng = np.random.default_rng(n_obs)
    boxes = np.zeros((n_obs, 10, n), np.float32)
    boxes[:, 0:3] = rng.uniform(-3, 3, (n_obs, 3, n))
    boxes[:, 3:6] = rng.choice([0.05, 0.1, 0.2], (n_obs, 3, n))
    boxes[::2, 3:6] = np.array([4.0, 0.05, 4.0], np.float32)[None, :, None] / np.sqrt(n_obs)
    q = rng.normal(size=(n_obs, 4, n))
    boxes[:, 6:10] = q / np.linalg.norm(q, axis=1, keepdims=True)
    st = np.zeros((13, n), np.float32)
    st[0:3], st[6] = rng.uniform(-3, 3, (3, n)), 1.0
    fl = Fleet(n, n_obstacles=n_obs, n_hexa=1300, n_octo=1300, dt=1e-30, seed=4)
    fl.set_obstacles(boxes)
    fl.set_state(st)
    fl.step(steps)
    hit = fl.events()[0].cpu().numpy() != 0
    fl.close()
    margin = box_margin(st[0:3].astype(np.float64), boxes.astype(np.float64), 0.2)
    sure = np.abs(margin) > 1e-4
    if steps == 1:
        np.testing.assert_array_equal(hit[sure], margin[sure] <= 0)
    else:                            # the second step tests the re-drawn vehicles too
        assert hit[sure & (margin <= 0)].all() and not hit[sure & (margin > 0)].any()
    assert sure.mean() > 0.99 and 20 < hit.sum() < n
