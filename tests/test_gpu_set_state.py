"""ag_set_state copies small fleets' device arrays in one launch, 16 bytes at a
time where both ends are aligned: any size and alignment must arrive whole, as
through the host copies."""
import numpy as np
import pytest
import torch

from paper_2305_16510_gb300 import _abi
from paper_2305_16510_gb300.fleet import Fleet

pytestmark = pytest.mark.gpu


def _shifted(a, dtype, words):
    """The array on the device, starting `words` 4-byte words after a 16-byte boundary."""
    flat = torch.zeros(a.size + words, dtype=dtype, device="cuda")
    flat[words:] = torch.from_numpy(a.reshape(-1)).cuda()
    return flat[words:].view(a.shape)


@pytest.mark.parametrize("with_epoch", [True, False])
@pytest.mark.parametrize("n", [1, 2, 3, 255, 1025, 70001, (1 << 19) + 1])
def test_set_state_from_device_arrays_of_any_alignment(n, with_epoch):
    rng = np.random.default_rng(n)
    state, motors = rng.normal(size=(13, n)).astype(np.float32), rng.normal(size=(8, n)).astype(np.float32)
    epoch = rng.integers(1, 1000, n).astype(np.int32)
    fl = Fleet(n)
    for shift in (0, 1, 2, 4):
        fl.set_state(np.zeros((13, n), np.float32), np.zeros((8, n), np.float32), np.zeros(n, np.int32))
        fl.synchronize()
        s, m, e = (_shifted(a, t, shift) for a, t in ((state, torch.float32), (motors, torch.float32), (epoch, torch.int32)))
        assert s.is_contiguous()
        _abi.ag_set_state(fl.ctx, s, m, e if with_epoch else None)
        np.testing.assert_array_equal(fl.state().cpu().numpy(), state)
        np.testing.assert_array_equal(fl.motors().cpu().numpy(), motors)
        np.testing.assert_array_equal(fl.epoch().cpu().numpy(), epoch if with_epoch else np.zeros(n, np.int32))
    fl.close()


@pytest.mark.parametrize("n", [8191, 600_001, (1 << 20) + 3, (1 << 23) + 1])
def test_set_state_around_the_lines_between_copies_and_kernel(n):
    """Blocks that take several turns; above 2^19 vehicles at an odd address and
    above 2^23 at any the copies serve."""
    torch.manual_seed(n)
    for words in (0, 1):
        s = torch.rand(13 * n + words, device="cuda")[words:].view(13, n)
        m = torch.rand(8 * n + words, device="cuda")[words:].view(8, n)
        e = torch.randint(1, 1000, (n,), dtype=torch.int32, device="cuda")
        fl = Fleet(n)
        _abi.ag_set_state(fl.ctx, s, m, e)
        assert torch.equal(fl.state(), s) and torch.equal(fl.motors(), m) and torch.equal(fl.epoch(), e)
        fl.close()
