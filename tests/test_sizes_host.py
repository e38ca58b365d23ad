"""Sizes of device arrays, checked on the host: products of counts that the
interface admits may exceed 64 bits, and must then be refused, not wrapped to a
small allocation that the kernels would write past."""
import subprocess

from paper_2305_16510_gb300 import build

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
