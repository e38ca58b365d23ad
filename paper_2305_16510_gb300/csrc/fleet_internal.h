// fleet_internal.h — launch interface between the C-ABI layer and the kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "ag.h"
#include "fleet_device.cuh"
#include "reset_sampler.cuh"

namespace agk {

// NVTX range over a host-side span (a C-ABI call's checks and enqueueing, a
// serving chunk), so a profiler's timeline names what issued each kernel.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// The grouping order. Windows of kOrderWindow consecutive environments are each
// partitioned by key (rotor type, command mode); a key's run of slots starts at
// a multiple of 32, so that no warp holds two keys, and the slots between runs
// hold kNoEnv. A window has room for four keys per rotor type in it, each run
// rounded up: under 1 % more slots than environments, but for the two windows
// in which the type may change.
constexpr uint32_t kOrderWindow = 16384;
constexpr uint32_t kNoEnv = 0xFFFFFFFFu;
struct OrderLayout {
  uint32_t n, n_quad, n_hexa;
  static constexpr __host__ __device__ uint32_t room(uint32_t count, uint32_t types) {
    return (count + 31u * 4u * types) / 32u * 32u;
  }
  __host__ __device__ uint32_t count(uint32_t w) const {
    const uint32_t lo = w * kOrderWindow;
    return n - lo < kOrderWindow ? n - lo : kOrderWindow;
  }
  __host__ __device__ uint32_t types(uint32_t w) const {
    const uint32_t lo = w * kOrderWindow, hi = lo + count(w), octo = n_quad + n_hexa;
    return (lo < n_quad ? 1u : 0u) + ((lo > n_quad ? lo : n_quad) < (hi < octo ? hi : octo) ? 1u : 0u) +
           ((lo > octo ? lo : octo) < hi ? 1u : 0u);
  }
  __host__ __device__ uint32_t slots(uint32_t w) const { return room(count(w), types(w)); }
  __host__ __device__ uint32_t windows() const { return (n + kOrderWindow - 1) / kOrderWindow; }
  // First slot of window w.
  __host__ __device__ uint32_t base(uint32_t w) const {
    const uint32_t v1 = n_quad / kOrderWindow, v2 = (n_quad + n_hexa) / kOrderWindow, one = room(kOrderWindow, 1);
    return w * one + (v1 < w ? slots(v1) - one : 0u) + (v2 != v1 && v2 < w ? slots(v2) - one : 0u);
  }
  // Slots of the fleet (a multiple of 32).
  __host__ __device__ uint32_t total() const { return base(windows() - 1) + slots(windows() - 1); }
};

// What a call counts, side by side so that one memset clears it.
struct CallCounts {
  unsigned long long tests;  // collision tests of the last fused call
  uint32_t resets;           // length of the reset list
};

// Device buffers of one fleet (all structure-of-arrays over n environments).
struct FleetBuffers {
  float* state;        // [13][n]  p, v, q, Omega
  float* motors;       // [8][n]   rotor thrusts
  float* body;         // [4][n]   m, Jxx, Jyy, Jzz
  uint8_t* modes;      // [n]
  float* targets;      // [4][n]
  float* boxes;        // [n_obs][10][n] centre, half-extents, quaternion: the caller's array of the
                       // allocation-free step; a context keeps the box records below instead
  float4* box_bound;   // [n_obs][n]    (centre, radius of the circumscribed sphere)
  float4* box_rest;    // [n_obs][n][2] (half-extents, q_w) (q_x, q_y, q_z, 0)
  uint32_t* epoch;     // [n]
  uint8_t* collided;   // [n]     hit a box during the last call
  uint32_t* reset_ids; // [n]     compact list of envs reset during the last call
  uint32_t* n_reset;   // [1]     length of that list
  // scratch of the unfused path (one launch per stage)
  float* cmd;          // [4][n]  commanded wrench
  float* wrench;       // [4][n]  realised wrench
  uint32_t* resets;    // [n]     resets of this call per env
  uint8_t* hits;       // [n]     collision of the current step
  uint32_t* order;     // [n_slots] thread slot -> env, grouped by rotor type and mode, kNoEnv in the
                       // padding (NULL = identity over n slots)
  const BoxRandDev* box_rand;  // [n_obs] obstacle re-draw on reset (NULL = boxes keep their poses)
  CallCounts* counts;  // [1] a context's counts; n_reset points into it (NULL for the other users)
  uint32_t n, n_quad, n_hexa, n_octo, n_obs;
  uint32_t n_slots;    // thread slots of order (OrderLayout::total)
};

// Launch constants of a configuration: gains, FP64-computed allocation
// matrices of the three rotor types, substep length, motor-lag factor,
// drag, squared collision radius, thrust limit and the reset key.
StepParams step_params_for(const ag_config& c, uint64_t seed);

// Launches return cudaGetLastError() of their launch.
cudaError_t launch_fused_step(const FleetBuffers& fb, const StepParams& P, int integrator, int n_steps,
                              int substeps, cudaStream_t st);
cudaError_t launch_reset(const FleetBuffers& fb, const uint8_t* mask, uint32_t seed_lo, uint32_t seed_hi,
                         cudaStream_t st);
// The controller alone: fb.cmd[4][n] = commanded (f, M) of every environment
// at fb.state (the unfused path's controller stage).
cudaError_t launch_controller(const FleetBuffers& fb, const StepParams& P, cudaStream_t st);
cudaError_t launch_plain_step(const FleetBuffers& fb, const StepParams& P, int integrator, int n_steps,
                              int substeps, cudaStream_t st);

// Builds fb.order from the current modes and rotor types (one launch).
cudaError_t launch_build_order(const FleetBuffers& fb, cudaStream_t st);

// Box records of boxes k0 .. k0 + count - 1 from the layout of ag_set_obstacles
// (row f of box k0 + j at src[(j * 10 + f) * pitch + env]), and back (pitch n).
cudaError_t launch_pack_boxes(const FleetBuffers& fb, const float* src, size_t pitch, uint32_t k0, uint32_t count,
                              cudaStream_t st);
cudaError_t launch_unpack_boxes(const FleetBuffers& fb, float* dst, uint32_t k0, uint32_t count, cudaStream_t st);

// Device memory for rows of boxes on their way to or from memory that a kernel
// does not reach in place: at least one box's rows, better all of them.
struct BoxStage {
  float* rows;
  size_t bytes;
  uint32_t boxes(uint32_t n) const {
    const size_t fit = bytes / (10 * sizeof(float) * n);
    return fit < 1 ? 1u : fit > 64 ? 64u : (uint32_t)fit;
  }
};
// All boxes of fb from any memory (rows of `pitch` elements), and to any memory
// (pitch n), as many at a time as the stage holds. One at a time, 64 boxes of
// 1,000 environments take 864 us to read and 690 to set, together 30 and 354; the
// eight requests of a batch with 16 boxes from host memory 3,047 us against 1,235.
cudaError_t upload_boxes(const FleetBuffers& fb, const float* boxes, size_t pitch, const BoxStage& stage, cudaStream_t st);
cudaError_t download_boxes(const FleetBuffers& fb, float* boxes, const BoxStage& stage, cudaStream_t st);
// A stage of several boxes, made when the first transfer wants it (cudaMalloc of
// 160 MB takes 0.5 ms, which a program that sets its boxes from device memory does
// not pay); NULL if the device has no room for it.
float* alloc_box_stage(size_t bytes);

// Bytes of the box records of n envs with n_obs boxes each.
inline size_t box_record_bytes(size_t n, size_t n_obs) { return n * n_obs * 3 * sizeof(float4); }

// Launch choices of the fused kernel. Defaults: mode-grouped order, the
// block size (from 64, 128, 96, 32) with the most resident warps per SM by
// the occupancy calculator (block = 0 here), and collision tests skipped
// while a vehicle provably cannot reach a box. Tuning overrides (read at each
// launch): AG_FUSED_ORDER=identity runs env i in slot i (the ungrouped
// ablation), AG_FUSED_BLOCK=32..128 (multiple of 32) sets the block size,
// AG_FUSED_SKIP=0 tests every box at every step (same results, the reference
// the skip and the bounding spheres are checked against).
struct FusedTuning { bool sorted; int block; bool skip; };
FusedTuning fused_tuning_from_env();

}  // namespace agk
