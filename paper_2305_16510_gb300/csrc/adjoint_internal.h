// adjoint_internal.h — launch interface of the differentiable rollout.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "fleet_device.cuh"

namespace agk {

// float4 words of one tape entry of one vehicle.
constexpr int kTapeWords = 4;

// Whether a tape of `entries` entries with `slots` columns keeps a context that
// holds `other` bytes beside it within `budget` (0 = no limit). 2^30 steps of
// 2^28 vehicles are more bytes than 64 bits hold, so nothing is multiplied out
// before it is known to fit.
inline bool tape_within_budget(uint64_t budget, size_t other, size_t entries, size_t slots) {
  return budget == 0 || (other <= budget && entries <= (budget - other) / (kTapeWords * slots * sizeof(float4)));
}

// Device buffers of one recorded rollout and its adjoint. Arrays marked
// "slot" have n_slots columns, one per thread slot (environment order[slot],
// none in the padding); the others are indexed by environment. With full_tape
// the tape holds the entries of every step and the end state; else it holds one
// segment's K entries, and checkpoint s holds the state (13 rows) and motors (8
// rows) at step s * K.
struct AdjointBuffers {
  float* state;                // [13][n] fleet state (advanced by the record)
  float* motors;               // [8][n]
  const float* body;           // [4][n]
  const uint8_t* modes;        // [n] command mode per env (values above 3 act as a wrench)
  const float* targets;        // [4][n] command targets
  const uint32_t* order;       // [n_slots] thread slot -> environment, grouped by rotor type and mode
  const float* goal_in;        // [3][n] the record's goals (the caller's array, or p_goal)
  float* p_goal;               // [3][n] kept for the sweep, written by the record
  float* ckpt;                 // [S][21][n] (NULL with full_tape)
  float4* tape;                // [n_steps + 1][4] (full_tape) or [K][4], slot
  float* inv_q0;               // slot: 1 / |q_0| of the given initial quaternion
  float* loss;                 // [n]
  uint8_t* saturated;          // [n] some motor hit a clamp during the record
  const float* loss_weights;   // [n] upstream gradient of each env's loss (NULL = 1)
  float* grad_x0;              // [13][n] (NULL = not wanted, as the next three)
  float* grad_gains_env;       // [12][n]
  float* grad_targets;         // [4][n]
  float* grad_gains;           // [12]
  float* partial;              // [12][n_slots / 32]: one sum per warp
  uint32_t n, n_slots, n_quad, n_hexa, n_octo;
  int n_steps, K;
  int full_tape;               // 1: the record wrote the whole horizon's tape
  float w_pos, w_omega;
};

cudaError_t launch_record(const AdjointBuffers& ab, const StepParams& P, cudaStream_t st);
cudaError_t launch_adjoint(const AdjointBuffers& ab, const StepParams& P, cudaStream_t st);

}  // namespace agk
