"""Sizes of device arrays, checked on the host: products of counts that the
interface admits may exceed 64 bits, and must then be refused, not wrapped to a
small allocation that the kernels would write past."""
import subprocess

import pytest

from paper_2305_16510_gb300 import _abi, build

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>
static size_t asked;
static cudaError_t record_malloc(void** p, size_t bytes) { asked = bytes; *p = (void*)256; return cudaSuccess; }
#define cudaMalloc record_malloc
#include "adjoint_internal.h"
#include "ctx_internal.h"

int main() {
  ag_ctx ctx{};
  float* f = nullptr;
  float4* v = nullptr;
  // a whole-horizon tape (steps and slots as below) and checkpoints of every step
  const size_t slots = 270008320, full = 1067487017ull + 1;
  int bad = 0;
  asked = 0;
  bad += agh::alloc(&ctx, &v, full * agk::kTapeWords * slots) != cudaErrorMemoryAllocation || asked != 0;
  bad += agh::alloc(&ctx, &f, (1ull << 30) * 21 * slots) != cudaErrorMemoryAllocation || asked != 0;
  bad += agh::alloc(&ctx, &f, SIZE_MAX / sizeof(float) + 1) != cudaErrorMemoryAllocation || asked != 0;
  bad += ctx.bytes != 0;
  bad += agh::alloc(&ctx, &f, 1000) != cudaSuccess || asked != 4000 || ctx.bytes != 4000;
  // the budget: 12.8 GB is what the bytes of that tape wrap to
  const uint64_t budget = 40ull << 30;
  bad += agk::tape_within_budget(budget, 0, full, slots);
  bad += agk::tape_within_budget(budget, budget + 1, 1, 32);   // other buffers beyond it already
  bad += !agk::tape_within_budget(0, 1ull << 60, full, slots);  // no limit: the allocation decides
  const size_t entry = agk::kTapeWords * 96 * sizeof(float4);
  bad += !agk::tape_within_budget(1000 + 5 * entry, 1000, 5, 96) || agk::tape_within_budget(999 + 5 * entry, 1000, 5, 96);
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_sizes_beyond_64_bits_do_not_fit(tmp_path):
    src = tmp_path / "sizes.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "sizes"
    r = subprocess.run([build._nvcc(), "-std=c++17", f"-I{build.INCLUDE}", f"-I{build.CSRC}", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert (r.returncode, r.stdout.strip()) == (0, "0")


def _order_slots(n, n_quad, n_hexa):
    """Slots of the grouping order: windows of 16,384 environments, each with
    room for four runs per rotor type in it, rounded up to 32 slots each."""
    total, octo = 0, n_quad + n_hexa
    for lo in range(0, n, 16384):
        hi = min(lo + 16384, n)
        types = (lo < n_quad) + (max(lo, n_quad) < min(hi, octo)) + (max(lo, octo) < hi)
        total += (hi - lo + 31 * 4 * types) // 32 * 32
    return total


@pytest.mark.parametrize("n_obs", [0, 1, 7])
@pytest.mark.parametrize("n,n_hexa,n_octo", [(1, 0, 0), (1000, 0, 0), (1000, 300, 200), (16385, 0, 1), (100_000, 33_000, 1)])
def test_budget_counts_everything_a_context_allocates(n, n_hexa, n_octo, n_obs):
    """state 13, motors 8, body, targets and the wrench scratch 4 rows each;
    epoch, reset ids and reset counts; modes, collided, hits and mask bytes;
    the order with its padding; box records and one box's staging; two
    counters and the check counter."""
    c = _abi.ag_config_default()
    c.n_envs, c.n_quad, c.n_hexa, c.n_octo, c.n_obstacles = n, n - n_hexa - n_octo, n_hexa, n_octo, n_obs
    need = (n * (33 * 4 + 3 * 4 + 4) + 4 * _order_slots(n, c.n_quad, n_hexa) + n * n_obs * 48 +
            (40 * n if n_obs else 0) + 16 + 4)
    c.hbm_budget_bytes = need - 1
    with pytest.raises(_abi.AgError) as e:
        _abi.ag_create(c)
    assert e.value.status == _abi.AG_ERR_OOM and str(need) in str(e.value)
    c.hbm_budget_bytes = need            # enough: what comes next is the device
    try:
        _abi.ag_destroy(_abi.ag_create(c))
    except _abi.AgError as err:
        assert err.status == _abi.AG_ERR_CUDA
