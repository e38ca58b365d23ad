// fleet_kernels.cu — the fused fleet-step kernel, the reset kernel and the
// unfused (one launch per stage) comparison path.
//
// Fused step (the hot path): one thread owns one environment for a whole
// launch of n_steps steps. Its 13 state words, motor thrusts, body
// parameters and command live in registers across every substep; its boxes
// are read only when a collision test runs (the first step, then only while
// the vehicle may be within reach of a box); state and command are read at
// the start and written at the end of the launch (coalesced structure-of-arrays rows).
// Collision resets happen in registers; the reset list is built with one
// __ballot_sync + __popc prefix and one atomicAdd per warp.
#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include <cuda_runtime.h>

#include "fleet_internal.h"
#include "fleet_sim.cuh"
#include "reset_sampler.cuh"

namespace agk {
namespace {

// Thread slot i of the launch simulates environment order[i] (a permutation
// that groups environments of equal rotor count and command mode, so the
// mode branches of the controller are warp-uniform), or environment i when
// order is NULL. A collision test that cannot hit is skipped (simulate_cmd),
// so tests are rare after the first step; a test reads the environment's box
// records (EnvBoxes). Threads of one command mode run the loop compiled for
// that mode (simulate). With boxes the bound of 4 blocks of 128 threads
// per SM holds the kernel under 128 registers, 4 warps per SM sub-partition
// (16 per SM); a bound of 3 (140 registers, 12 warps per SM) measured
// slower.
// Without obstacles the kernel stays within 128 registers. A quad-only
// semi-implicit-Euler fleet without obstacles needs about 70 (no spills),
// and its bound of 7 blocks per SM lets a 131,072-vehicle fleet run in one
// wave; fleets with hexa and octo rotors keep the looser bound, which
// measured faster for them.
// SINGLE: a launch of one step among boxes, where every vehicle tests and none
// needs a clearance. It has one loop body for all modes, like the task step, and
// loads spheres and marked boxes in groups (EnvBoxesT<true, true>), for which the
// loops of the many-step kernel leave no registers. Among walls, whose spheres
// exclude nothing (half-extents 5 x 5 x 0.05 m), 250,007 quads x 8 take 40.9 us a
// call instead of 47.7 and x 30 66.2 instead of 83.8; among 16 boxes of U[0.1, 1] m
// 29.5 instead of 30.8.
template <int INTEG, bool QUAD_ONLY, bool DRAG, bool BOXES, bool SINGLE>
__global__ void __launch_bounds__(128, !BOXES && QUAD_ONLY && INTEG == kIntegSIE ? 7 : 4)
    k_fused_step(FleetBuffers fb, StepParams P, int n_steps, int substeps) {
  const uint32_t slot = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t env = fb.order ? (slot < fb.n_slots ? fb.order[slot] : kNoEnv) : slot;
  const bool active = env < fb.n;
  uint32_t resets = 0, tests = 0;
  bool any_hit = false;
  if (active) {
    const int nrot = QUAD_ONLY ? 4 : rotor_count(fb, env);
    const std::conditional_t<BOXES, EnvBoxesT<SINGLE, SINGLE>, NoBoxSource> boxes(fb, env);
    const int n_obs = BOXES ? (int)fb.n_obs : 0;
    if (SINGLE) n_steps = 1;
    if (nrot == 4)
      simulate<4, INTEG, DRAG, !SINGLE>(fb, P, env, n_steps, substeps, n_obs, boxes, P.seed_lo, P.seed_hi, resets, any_hit, tests);
    else if (nrot == 6)
      simulate<6, INTEG, DRAG, !SINGLE>(fb, P, env, n_steps, substeps, n_obs, boxes, P.seed_lo, P.seed_hi, resets, any_hit, tests);
    else
      simulate<8, INTEG, DRAG, !SINGLE>(fb, P, env, n_steps, substeps, n_obs, boxes, P.seed_lo, P.seed_hi, resets, any_hit, tests);
    fb.collided[env] = any_hit ? 1 : 0;
  }
  if (!BOXES) {  // nothing can be reset: the counts are cleared here, not by a memset before the launch
    if (slot == 0) *fb.counts = CallCounts{0, 0};
    return;
  }
  append_compact(resets > 0u, env, fb.reset_ids, &fb.counts->resets);
  const unsigned t = __reduce_add_sync(0xFFFFFFFFu, tests);  // one atomic per warp
  if ((threadIdx.x & 31u) == 0u && t) atomicAdd(&fb.counts->tests, (unsigned long long)t);
}

// Grouping order: key = rotor-type index * 4 + mode (12 keys). Each window of
// 16,384 environments is stably partitioned by key, every key's run of slots
// starting at a multiple of 32 (OrderLayout): a warp then holds one key and the
// controller's mode branches are warp-uniform, and since a window's envs are
// loaded by blocks that run at the same time, the sectors their gathers share
// are served from L2 instead of being fetched again from DRAM. With runs that
// were not padded, one warp per key boundary ran two modes' code in turn, and
// launches of one wave waited for it (131,072 quads of two modes x 100 steps:
// 127 us a pass against 121; 1,000 quads' gradient 491 us against 412). A
// window of 4,096 needs four times the padding (8 % with three rotor types,
// which cost a 4M mixed fleet 0.9 %).
// One block per window. Each warp takes a contiguous share of the window's
// environments, 32 at a time, and ranks them by key (__match_any_sync, one
// add per key and 32 environments); a scan over the warps gives every warp its
// place in each key's run, and the environments go to their slots. All ROUNDS
// modes of a thread are requested, and all matches made, before any is counted:
// a kernel that asked for each mode as it came to it, twice, took 18.6 us a call of
// ag_set_commands for 16,384 to 1M quads, this one 12.5 to 14.5. Fleets of up to
// 1,024 and 4,096 environments take 1 and 4 rounds; with 16 they wait 2 us longer.
constexpr int kOrderThreads = 1024, kOrderWarps = kOrderThreads / 32;
constexpr int kOrderRounds = kOrderWindow / kOrderThreads;  // environments per thread of a whole window

__host__ __device__ inline OrderLayout order_layout(const FleetBuffers& fb) { return {fb.n, fb.n_quad, fb.n_hexa}; }

__device__ __forceinline__ uint32_t order_key(const FleetBuffers& fb, uint32_t i) {
  const int nrot = rotor_count(fb, i);
  const uint32_t m = fb.modes[i] > 3 ? 3u : fb.modes[i];
  return (uint32_t)(nrot == 4 ? 0 : (nrot == 6 ? 1 : 2)) * 4u + m;
}

template <int ROUNDS>
__global__ void __launch_bounds__(kOrderThreads) k_order_window(FleetBuffers fb) {
  __shared__ uint32_t place[kOrderWarps][13];  // counts (the last: of no environment), then the warp's place in each key's run
  __shared__ uint32_t run[12];                 // length, then the first slot of each key's run
  const OrderLayout layout = order_layout(fb);
  const uint32_t first = blockIdx.x * kOrderWindow, count = layout.count(blockIdx.x), slots = layout.slots(blockIdx.x);
  uint32_t* const order = fb.order + layout.base(blockIdx.x);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const uint32_t share = (count + kOrderThreads - 1) / kOrderThreads * 32u;  // environments per warp
  const uint32_t lo = warp * share, hi = min(lo + share, count);
  uint32_t key[ROUNDS], rank[ROUNDS];  // of environment lo + 32 j + lane in its warp's share
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const uint32_t i = lo + 32u * j + lane;
    key[j] = i < hi ? order_key(fb, first + i) : 12u;
  }
  for (uint32_t k = threadIdx.x; k < slots; k += kOrderThreads) order[k] = kNoEnv;
  if (lane < 13) place[warp][lane] = 0;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) rank[j] = __match_any_sync(0xFFFFFFFFu, key[j]);
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const unsigned same = rank[j];
    const uint32_t before = place[warp][key[j]];
    __syncwarp();
    rank[j] = before + __popc(same & ((1u << lane) - 1u));
    if ((int)lane == __ffs(same) - 1) place[warp][key[j]] = before + __popc(same);
    __syncwarp();
  }
  __syncthreads();
  if (warp < 12) {  // warp k: exclusive scan of key k's counts over the warps
    const uint32_t own = place[lane][warp];
    uint32_t sum = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, sum, d);
      if ((int)lane >= d) sum += up;
    }
    place[lane][warp] = sum - own;
    if (lane == 31) run[warp] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t at = 0;
    for (int k = 0; k < 12; ++k) {
      const uint32_t length = run[k];
      run[k] = at;
      at += (length + 31u) & ~31u;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ROUNDS; ++j)
    if (key[j] < 12u) order[run[key[j]] + place[warp][key[j]] + rank[j]] = first + lo + 32u * j + lane;
}

// Box records k0 .. from the caller's rows and back: thread (env, box).
__global__ void __launch_bounds__(256) k_pack_boxes(FleetBuffers fb, const float* __restrict__ src, size_t pitch,
                                                    uint32_t k0) {
  const uint32_t env = blockIdx.x * blockDim.x + threadIdx.x;
  if (env >= fb.n) return;
  float v[10];
#pragma unroll
  for (int f = 0; f < 10; ++f) v[f] = src[((size_t)blockIdx.y * 10 + f) * pitch + env];
  pack_box(fb, k0 + blockIdx.y, env, v);
}

__global__ void __launch_bounds__(256) k_unpack_boxes(FleetBuffers fb, float* __restrict__ dst, uint32_t k0) {
  const uint32_t env = blockIdx.x * blockDim.x + threadIdx.x;
  if (env >= fb.n) return;
  const size_t at = (size_t)(k0 + blockIdx.y) * fb.n + env;
  const float4 b = fb.box_bound[at], h = fb.box_rest[2 * at], q = fb.box_rest[2 * at + 1];
  const float v[10] = {b.x, b.y, b.z, h.x, h.y, h.z, h.w, q.x, q.y, q.z};
#pragma unroll
  for (int f = 0; f < 10; ++f) dst[((size_t)blockIdx.y * 10 + f) * fb.n + env] = v[f];
}

// ag_reset: resample masked environments, clear collided flags, list them.
__global__ void __launch_bounds__(256) k_reset(FleetBuffers fb, const uint8_t* mask, uint32_t seed_lo,
                                               uint32_t seed_hi) {
  const uint32_t env = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t n = fb.n;
  const bool active = env < n;
  const bool flag = active && (mask == nullptr || mask[env] != 0);
  if (flag) reset_env(fb, env, seed_lo, seed_hi);
  if (active) fb.collided[env] = 0;
  append_compact(flag, env, fb.reset_ids, fb.n_reset);
}

// ------------------------------------------------ unfused comparison path --
__global__ void __launch_bounds__(256) k_plain_controller(FleetBuffers fb, StepParams P) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= fb.n) return;
  const uint32_t n = fb.n;
  VState s = load_state(fb.state, n, i);
  normalize(s.q);
  V3 b3;
  Wrench4 c = controller(s, load_command(fb, i), load_body(fb.body, n, i), P, b3);
  fb.cmd[0 * n + i] = c.f; fb.cmd[1 * n + i] = c.mx; fb.cmd[2 * n + i] = c.my; fb.cmd[3 * n + i] = c.mz;
}

template <int NROT>
__device__ __forceinline__ void plain_allocate_one(const FleetBuffers& fb, const StepParams& P, uint32_t i) {
  const uint32_t n = fb.n;
  float u[NROT];
#pragma unroll
  for (int k = 0; k < NROT; ++k) u[k] = fb.motors[k * n + i];
  Wrench4 c = {fb.cmd[0 * n + i], fb.cmd[1 * n + i], fb.cmd[2 * n + i], fb.cmd[3 * n + i]};
  Wrench4 W = allocate<NROT>(c, u, P);
#pragma unroll
  for (int k = 0; k < NROT; ++k) fb.motors[k * n + i] = u[k];
  fb.wrench[0 * n + i] = W.f; fb.wrench[1 * n + i] = W.mx; fb.wrench[2 * n + i] = W.my; fb.wrench[3 * n + i] = W.mz;
}

__global__ void __launch_bounds__(256) k_plain_allocate(FleetBuffers fb, StepParams P) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= fb.n) return;
  const int nrot = rotor_count(fb, i);
  if (nrot == 4) plain_allocate_one<4>(fb, P, i);
  else if (nrot == 6) plain_allocate_one<6>(fb, P, i);
  else plain_allocate_one<8>(fb, P, i);
}

template <int INTEG, bool DRAG>
__global__ void __launch_bounds__(256) k_plain_integrate(FleetBuffers fb, StepParams P) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= fb.n) return;
  const uint32_t n = fb.n;
  VState s = load_state(fb.state, n, i);
  Wrench4 W = {fb.wrench[0 * n + i], fb.wrench[1 * n + i], fb.wrench[2 * n + i], fb.wrench[3 * n + i]};
  integrate<INTEG, DRAG>(s, body_z(s.q), W, load_body(fb.body, n, i), P);
  store_state(fb.state, n, i, s);
}

// Collision test of every environment against its boxes: every box of the
// caller's rows (the allocation-free step), or the context's records, spheres
// first as in the fused step; the per-env hit byte goes to `collided_now`.
__global__ void __launch_bounds__(256) k_plain_collide(FleetBuffers fb, StepParams P, uint8_t* collided_now) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= fb.n) return;
  const uint32_t n = fb.n;
  V3 p = {fb.state[0 * n + i], fb.state[1 * n + i], fb.state[2 * n + i]};
  bool hit = false;
  if (fb.boxes) {
    for (uint32_t k = 0; k < fb.n_obs; ++k) {
      const float* bx = fb.boxes + (size_t)k * 10 * n + i;
      hit |= touches(P.r2, box_dist2(p, V3{bx[0], bx[n], bx[2 * n]}, V3{bx[3 * n], bx[4 * n], bx[5 * n]},
                                     Q4{bx[6 * n], bx[7 * n], bx[8 * n], bx[9 * n]}));
    }
  } else {
    float clearance2;
    hit = EnvBoxesT<true, true>(fb, i).any_hit(p, sqrtf(P.r2), P.r2, (int)fb.n_obs, kBoxSlack, false, clearance2);
  }
  collided_now[i] = hit ? 1 : 0;
}

__global__ void __launch_bounds__(256) k_plain_reset_hits(FleetBuffers fb, StepParams P, const uint8_t* collided_now) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= fb.n || collided_now[i] == 0) return;
  const uint32_t n = fb.n;
  const uint32_t epoch = fb.epoch[i] + 1u;
  fb.epoch[i] = epoch;
  fb.resets[i] += 1u;
  fb.collided[i] = 1;
  ResetValues r = draw_reset(P.seed_lo, P.seed_hi, i, epoch);
  float* st = fb.state;
  st[0 * n + i] = r.p[0]; st[1 * n + i] = r.p[1]; st[2 * n + i] = r.p[2];
  st[3 * n + i] = r.v[0]; st[4 * n + i] = r.v[1]; st[5 * n + i] = r.v[2];
  st[6 * n + i] = r.q[0]; st[7 * n + i] = r.q[1]; st[8 * n + i] = r.q[2]; st[9 * n + i] = r.q[3];
  st[10 * n + i] = 0.f; st[11 * n + i] = 0.f; st[12 * n + i] = 0.f;
  const int nrot = rotor_count(fb, i);
  const float hv = hover_per_motor(fb.body[i], nrot);
  for (int k = 0; k < nrot; ++k) fb.motors[k * n + i] = hv;
  if (fb.box_rand) redraw_boxes(fb, i, epoch, P.seed_lo, P.seed_hi);
}

__global__ void __launch_bounds__(256) k_plain_compact(FleetBuffers fb) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool pred = i < fb.n && fb.resets[i] > 0u;
  append_compact(pred, i, fb.reset_ids, fb.n_reset);
}

template <int INTEG, bool QUAD_ONLY, bool DRAG, bool BOXES, bool SINGLE>
cudaError_t launch_fused_b(const FleetBuffers& fb, const StepParams& P, int n_steps, int substeps, int B,
                           cudaStream_t st) {
  const auto kernel = k_fused_step<INTEG, QUAD_ONLY, DRAG, BOXES, SINGLE>;
  if (B == 0) {  // the block size with the most resident warps per SM (ties: the earlier candidate)
    int best = -1;
    for (int b : {64, 128, 96, 32}) {
      int blocks = 0;
      const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, b, 0);
      if (e != cudaSuccess) return e;
      if (blocks * b > best) { best = blocks * b; B = b; }
    }
    if (best <= 0) return cudaErrorInvalidConfiguration;
  }
  const uint32_t slots = fb.order ? fb.n_slots : fb.n;
  const unsigned grid = (slots + B - 1) / B;
  if (BOXES) {
    const cudaError_t e = cudaMemsetAsync(fb.counts, 0, sizeof(CallCounts), st);
    if (e != cudaSuccess) return e;
  }
  kernel<<<grid, B, 0, st>>>(fb, P, n_steps, substeps);
  return cudaGetLastError();
}

template <int INTEG, bool QUAD_ONLY, bool DRAG>
cudaError_t launch_fused_t(const FleetBuffers& fb, const StepParams& P, int n_steps, int substeps, int B,
                           cudaStream_t st) {
  if (fb.n_obs == 0) return launch_fused_b<INTEG, QUAD_ONLY, DRAG, false, false>(fb, P, n_steps, substeps, B, st);
  return n_steps == 1 ? launch_fused_b<INTEG, QUAD_ONLY, DRAG, true, true>(fb, P, n_steps, substeps, B, st)
                      : launch_fused_b<INTEG, QUAD_ONLY, DRAG, true, false>(fb, P, n_steps, substeps, B, st);
}

template <int INTEG>
cudaError_t launch_fused_i(const FleetBuffers& fb, const StepParams& P, int n_steps, int substeps, int B,
                           cudaStream_t st) {
  const bool quad_only = fb.n_quad == fb.n;
  const bool drag = P.drag != 0.f;
  if (quad_only)
    return drag ? launch_fused_t<INTEG, true, true>(fb, P, n_steps, substeps, B, st)
                : launch_fused_t<INTEG, true, false>(fb, P, n_steps, substeps, B, st);
  return drag ? launch_fused_t<INTEG, false, true>(fb, P, n_steps, substeps, B, st)
              : launch_fused_t<INTEG, false, false>(fb, P, n_steps, substeps, B, st);
}

}  // namespace

FusedTuning fused_tuning_from_env() {
  FusedTuning t;
  t.sorted = true;
  t.block = 0;
  t.skip = true;
  if (const char* v = std::getenv("AG_FUSED_ORDER")) t.sorted = std::strcmp(v, "identity") != 0;
  if (const char* v = std::getenv("AG_FUSED_SKIP")) t.skip = std::strcmp(v, "0") != 0;
  if (const char* v = std::getenv("AG_FUSED_BLOCK")) {
    int b = std::atoi(v);
    if (b >= 32 && b <= 128 && b % 32 == 0) t.block = b;
  }
  return t;
}

cudaError_t launch_fused_step(const FleetBuffers& fb_in, const StepParams& P, int integrator, int n_steps,
                              int substeps, cudaStream_t st) {
  const FusedTuning t = fused_tuning_from_env();
  FleetBuffers fb = fb_in;
  if (!t.sorted) fb.order = nullptr;
  StepParams Pl = P;
  if (!t.skip) Pl.exact_tests = 1;
  return integrator == kIntegRK4 ? launch_fused_i<kIntegRK4>(fb, Pl, n_steps, substeps, t.block, st)
                                 : launch_fused_i<kIntegSIE>(fb, Pl, n_steps, substeps, t.block, st);
}

cudaError_t launch_build_order(const FleetBuffers& fb, cudaStream_t st) {
  const auto kernel = fb.n <= kOrderThreads       ? k_order_window<1>
                      : fb.n <= 4 * kOrderThreads ? k_order_window<4>
                                                  : k_order_window<kOrderRounds>;
  kernel<<<order_layout(fb).windows(), kOrderThreads, 0, st>>>(fb);
  return cudaGetLastError();
}

cudaError_t launch_pack_boxes(const FleetBuffers& fb, const float* src, size_t pitch, uint32_t k0, uint32_t count,
                              cudaStream_t st) {
  k_pack_boxes<<<dim3((fb.n + 255) / 256, count), 256, 0, st>>>(fb, src, pitch, k0);
  return cudaGetLastError();
}

cudaError_t launch_unpack_boxes(const FleetBuffers& fb, float* dst, uint32_t k0, uint32_t count, cudaStream_t st) {
  k_unpack_boxes<<<dim3((fb.n + 255) / 256, count), 256, 0, st>>>(fb, dst, k0);
  return cudaGetLastError();
}

cudaError_t upload_boxes(const FleetBuffers& fb, const float* boxes, size_t pitch, const BoxStage& stage, cudaStream_t st) {
  const uint32_t most = stage.boxes(fb.n);
  for (uint32_t k = 0; k < fb.n_obs; k += most) {
    const uint32_t count = std::min(most, fb.n_obs - k);
    const float* src = boxes + (size_t)k * 10 * pitch;
    cudaError_t e = pitch == fb.n ? cudaMemcpyAsync(stage.rows, src, (size_t)count * 10 * fb.n * sizeof(float),
                                                    cudaMemcpyDefault, st)
                                  : cudaMemcpy2DAsync(stage.rows, fb.n * sizeof(float), src, pitch * sizeof(float),
                                                      fb.n * sizeof(float), (size_t)count * 10, cudaMemcpyDefault, st);
    if (e == cudaSuccess) e = launch_pack_boxes(fb, stage.rows, fb.n, k, count, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t download_boxes(const FleetBuffers& fb, float* boxes, const BoxStage& stage, cudaStream_t st) {
  const uint32_t most = stage.boxes(fb.n);
  for (uint32_t k = 0; k < fb.n_obs; k += most) {
    const uint32_t count = std::min(most, fb.n_obs - k);
    cudaError_t e = launch_unpack_boxes(fb, stage.rows, k, count, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(boxes + (size_t)k * 10 * fb.n, stage.rows, (size_t)count * 10 * fb.n * sizeof(float),
                          cudaMemcpyDefault, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

float* alloc_box_stage(size_t bytes) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // an allocation is no part of a capture
  cudaThreadExchangeStreamCaptureMode(&mode);
  float* p = nullptr;
  if (cudaMalloc((void**)&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return p;
}

cudaError_t launch_reset(const FleetBuffers& fb, const uint8_t* mask, uint32_t seed_lo, uint32_t seed_hi,
                         cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(fb.n_reset, 0, sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  const unsigned grid = (fb.n + 255) / 256;
  k_reset<<<grid, 256, 0, st>>>(fb, mask, seed_lo, seed_hi);
  return cudaGetLastError();
}

cudaError_t launch_controller(const FleetBuffers& fb, const StepParams& P, cudaStream_t st) {
  k_plain_controller<<<(fb.n + 255) / 256, 256, 0, st>>>(fb, P);
  return cudaGetLastError();
}

cudaError_t launch_plain_step(const FleetBuffers& fb, const StepParams& P, int integrator, int n_steps,
                              int substeps, cudaStream_t st) {
  const unsigned grid = (fb.n + 255) / 256;
  cudaError_t e = cudaMemsetAsync(fb.n_reset, 0, sizeof(uint32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(fb.resets, 0, sizeof(uint32_t) * fb.n, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(fb.collided, 0, fb.n, st);
  if (e != cudaSuccess) return e;
  uint8_t* hits = fb.hits;
  for (int step = 0; step < n_steps; ++step) {
    for (int ss = 0; ss < substeps; ++ss) {
      k_plain_controller<<<grid, 256, 0, st>>>(fb, P);
      k_plain_allocate<<<grid, 256, 0, st>>>(fb, P);
      const bool drag = P.drag != 0.f;
      if (integrator == kIntegRK4) {
        if (drag) k_plain_integrate<kIntegRK4, true><<<grid, 256, 0, st>>>(fb, P);
        else k_plain_integrate<kIntegRK4, false><<<grid, 256, 0, st>>>(fb, P);
      } else {
        if (drag) k_plain_integrate<kIntegSIE, true><<<grid, 256, 0, st>>>(fb, P);
        else k_plain_integrate<kIntegSIE, false><<<grid, 256, 0, st>>>(fb, P);
      }
    }
    if (fb.n_obs > 0) {
      k_plain_collide<<<grid, 256, 0, st>>>(fb, P, hits);
      k_plain_reset_hits<<<grid, 256, 0, st>>>(fb, P, hits);
    }
  }
  k_plain_compact<<<grid, 256, 0, st>>>(fb);
  return cudaGetLastError();
}

}  // namespace agk
