// task.cu — the reach-a-setpoint task around the fleet step.
//
// The paper trains policies that fly a multirotor to a goal setpoint through
// the attitude or the velocity command interface (Sec. I). One task step is
// one kernel launch: per environment the policy's action becomes its command,
// the fleet step runs (the fused step's per-vehicle loop: controller,
// allocation, integration, collision test and reset), and the step is scored;
// an episode that ended without a collision is re-drawn in place (a collision
// already re-drew its environment inside the step), and the observation of
// the state the policy sees next is written:
//   obs    = (p - g, v, q with w >= 0, Omega)                       [n][13]
//   reward = -crash after a collision, else -|p - g| - w_v |v| - w_omega |Omega|
//   done   = collided or |p - g| > max_dist or steps >= max_steps
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "fleet_sim.cuh"
#include "task_internal.h"

namespace agk {
namespace {

constexpr int kTaskBlock = 64;  // measured over 32 .. 256: 64 is best by about 1 %
constexpr int kObs = 13;

__device__ __forceinline__ float norm3(float x, float y, float z) { return sqrtf(fmaf(z, z, fmaf(y, y, x * x))); }

__device__ __forceinline__ V3 load_goal(const ReachArgs& a, uint32_t i) {
  const uint32_t n = a.fb.n;
  return {a.goals[i], a.goals[n + i], a.goals[2 * n + i]};
}

// obs = (p - g, v, q with w >= 0, Omega)
__device__ __forceinline__ void observe(const VState& s, V3 g, float* o) {
  const float sgn = s.q.w < 0.f ? -1.f : 1.f;
  o[0] = s.p.x - g.x; o[1] = s.p.y - g.y; o[2] = s.p.z - g.z;
  o[3] = s.v.x; o[4] = s.v.y; o[5] = s.v.z;
  o[6] = sgn * s.q.w; o[7] = sgn * s.q.x; o[8] = sgn * s.q.y; o[9] = sgn * s.q.z;
  o[10] = s.w.x; o[11] = s.w.y; o[12] = s.w.z;
}

// Reward, termination and in-place reset of environment i after its step
// (s: its state after the step; hit: it collided, and the step already
// re-drew it), then its observation into o[0..12].
__device__ __forceinline__ void reach_tail(const ReachArgs& a, uint32_t i, VState s, bool hit, uint32_t steps_before,
                                           V3 g, float* o) {
  const uint32_t steps = steps_before + 1u;
  const float dist = norm3(s.p.x - g.x, s.p.y - g.y, s.p.z - g.z);
  const float speed = norm3(s.v.x, s.v.y, s.v.z);
  const float rate = norm3(s.w.x, s.w.y, s.w.z);
  const bool end = hit || dist > a.max_dist || steps >= a.max_steps;
  a.reward[i] = hit ? -a.crash : -fmaf(a.w_omega, rate, fmaf(a.w_v, speed, dist));
  a.done[i] = end ? 1 : 0;
  a.steps[i] = end ? 0u : steps;
  if (end && !hit) {
    reset_env(a.fb, i, a.seed_lo, a.seed_hi);
    s = load_state(a.fb.state, a.fb.n, i);
  }
  observe(s, g, o);
}

// Coalesced write of the staged [kTaskBlock][13] observation rows, warp by
// warp: the rows of a warp's 32 environments are one contiguous slice of the
// stage and of obs, so each warp writes its own after a __syncwarp and no
// warp waits for the rest of the block.
__device__ __forceinline__ void write_obs(const ReachArgs& a, const float* stage) {
  __syncwarp();
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const size_t base = ((size_t)blockIdx.x * kTaskBlock + warp * 32u) * kObs;
  const size_t total = (size_t)a.fb.n * kObs;
  const float* ws = stage + warp * 32u * kObs;
#pragma unroll
  for (uint32_t t = lane; t < 32u * kObs; t += 32u)
    if (base + t < total) a.obs[base + t] = ws[t];
}

// The step itself for one airframe: action -> command t, one fleet step of
// `substeps` substeps from the vehicle's rows.
template <int NROT, int INTEG, bool DRAG, class Boxes>
__device__ __forceinline__ VState reach_fly(const ReachArgs& a, const StepParams& P, uint32_t i, float4 act, int mode,
                                            int substeps, int n_obs, const Boxes& boxes, float (&t)[4], bool& hit) {
  const VehicleRows<NROT> rows = load_vehicle<NROT>(a.fb, i);
  const float v[4] = {act.x, act.y, act.z, act.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] = fmaf(a.scale[k], fminf(fmaxf(v[k], -1.f), 1.f), a.offset[k]);
  const Command cm = prepare_command(mode, t[0], t[1], t[2], t[3]);
  uint32_t resets = 0, tests = 0;
  return simulate_cmd<NROT, INTEG, DRAG>(a.fb, P, i, rows, cm, 1, substeps, n_obs, boxes, a.seed_lo, a.seed_hi, resets,
                                         hit, tests);
}

// One task step of environment i = thread: actions -> commands, one fleet
// step (controller, allocation, integration, collision test and reset, as in
// the fused fleet step), then reach_tail. Every environment shares the task's
// command mode, so warps are mode-uniform without a grouping permutation.
// Without boxes the step is memory-latency bound: a bound of 12 blocks (24
// warps) per SM measured best (50.8 us a pass over 1,048,576 quads), against
// 10 (53.2), 14 (51.3), 16 (52.2, 64 registers) and 18 (53.3); with the state
// requested after the command's angles it took 57.4. RK4 is within 3 % of its best
// there: 1,048,576 quads x 4 substeps 73.9 us (10 blocks 72.7, 14 76.4), x 1 substep
// 49.4 (52.4, 54.2), mixed airframes x 4 80.6 (78.2, 79.6) and with drag 81.2 (78.6,
// 82.5), though those two kernels spill 40 and 72 bytes. With boxes 8 blocks (16
// warps, 128 registers).
template <int INTEG, bool QUAD_ONLY, bool DRAG, bool BOXES>
__global__ void __launch_bounds__(kTaskBlock, BOXES ? 8 : 12)
    k_reach_step(ReachArgs a, StepParams P, int substeps) {
  __shared__ float stage[kTaskBlock * kObs];  // odd row length: conflict-free
  const FleetBuffers& fb = a.fb;
  const uint32_t i = blockIdx.x * kTaskBlock + threadIdx.x;
  const uint32_t n = fb.n;
  if (i < n) {
    // everything the step reads from memory, requested up front
    const float4 act = reinterpret_cast<const float4*>(a.actions)[i];
    const V3 g = load_goal(a, i);
    const uint32_t steps_before = a.steps[i];
    const int mode = fb.modes[i];
    const int nrot = QUAD_ONLY ? 4 : rotor_count(fb, i);
    bool hit = false;
    VState s;
    float t[4];
    const std::conditional_t<BOXES, EnvBoxesT<true>, NoBoxSource> boxes(fb, i);
    const int n_obs = BOXES ? (int)fb.n_obs : 0;
    if (nrot == 4)
      s = reach_fly<4, INTEG, DRAG>(a, P, i, act, mode, substeps, n_obs, boxes, t, hit);
    else if (nrot == 6)
      s = reach_fly<6, INTEG, DRAG>(a, P, i, act, mode, substeps, n_obs, boxes, t, hit);
    else
      s = reach_fly<8, INTEG, DRAG>(a, P, i, act, mode, substeps, n_obs, boxes, t, hit);
    fb.collided[i] = hit ? 1 : 0;
    if (a.collided) a.collided[i] = hit ? 1 : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) fb.targets[k * n + i] = t[k];  // the commands, as ag_set_commands keeps them
    reach_tail(a, i, s, hit, steps_before, g, stage + threadIdx.x * kObs);
  }
  write_obs(a, stage);
}

__global__ void __launch_bounds__(kTaskBlock) k_reach_observe(ReachArgs a) {
  __shared__ float stage[kTaskBlock * kObs];
  const uint32_t i = blockIdx.x * kTaskBlock + threadIdx.x;
  if (i < a.fb.n) observe(load_state(a.fb.state, a.fb.n, i), load_goal(a, i), stage + threadIdx.x * kObs);
  write_obs(a, stage);
}

template <int INTEG, bool DRAG>
cudaError_t launch_step_t(const ReachArgs& a, const StepParams& P, int substeps, cudaStream_t st) {
  const unsigned grid = (a.fb.n + kTaskBlock - 1) / kTaskBlock;
  // with boxes a kernel for quads alone measured slower (36.9 us a pass against 35.6, 131,072 quads, 16 boxes)
  const auto kernel = a.fb.n_obs > 0           ? k_reach_step<INTEG, false, DRAG, true>
                      : a.fb.n_quad == a.fb.n ? k_reach_step<INTEG, true, DRAG, false>
                                              : k_reach_step<INTEG, false, DRAG, false>;
  kernel<<<grid, kTaskBlock, 0, st>>>(a, P, substeps);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_reach_step(const ReachArgs& a, const StepParams& P, int integrator, int substeps, cudaStream_t st) {
  const bool drag = P.drag != 0.f;
  if (integrator == kIntegRK4)
    return drag ? launch_step_t<kIntegRK4, true>(a, P, substeps, st) : launch_step_t<kIntegRK4, false>(a, P, substeps, st);
  return drag ? launch_step_t<kIntegSIE, true>(a, P, substeps, st) : launch_step_t<kIntegSIE, false>(a, P, substeps, st);
}

cudaError_t launch_reach_observe(const ReachArgs& a, cudaStream_t st) {
  k_reach_observe<<<(a.fb.n + kTaskBlock - 1) / kTaskBlock, kTaskBlock, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace agk
