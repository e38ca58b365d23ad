// fleet_sim.cuh — the per-vehicle loop shared by the fused kernels.
//
// Loading one environment into registers, running its steps (controller,
// allocation, integrator, collision test, in-register Philox reset) and
// storing it back; plus the warp-level compaction of reset ids. Used by the
// single-fleet fused kernel and by the multi-request serving kernel.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "fleet_device.cuh"
#include "fleet_internal.h"
#include "reset_sampler.cuh"

namespace agk {

__device__ __forceinline__ int rotor_count(const FleetBuffers& fb, uint32_t env) {
  if (env < fb.n_quad) return 4;
  if (env < fb.n_quad + fb.n_hexa) return 6;
  return 8;
}

__device__ __forceinline__ VState load_state(const float* st, uint32_t n, uint32_t i) {
  VState s;
  s.p = {st[0 * n + i], st[1 * n + i], st[2 * n + i]};
  s.v = {st[3 * n + i], st[4 * n + i], st[5 * n + i]};
  s.q = {st[6 * n + i], st[7 * n + i], st[8 * n + i], st[9 * n + i]};
  s.w = {st[10 * n + i], st[11 * n + i], st[12 * n + i]};
  return s;
}

__device__ __forceinline__ void store_state(float* st, uint32_t n, uint32_t i, const VState& s) {
  st[0 * n + i] = s.p.x; st[1 * n + i] = s.p.y; st[2 * n + i] = s.p.z;
  st[3 * n + i] = s.v.x; st[4 * n + i] = s.v.y; st[5 * n + i] = s.v.z;
  st[6 * n + i] = s.q.w; st[7 * n + i] = s.q.x; st[8 * n + i] = s.q.y; st[9 * n + i] = s.q.z;
  st[10 * n + i] = s.w.x; st[11 * n + i] = s.w.y; st[12 * n + i] = s.w.z;
}

__device__ __forceinline__ Body load_body(const float* bd, uint32_t n, uint32_t i) {
  return make_body(bd[0 * n + i], bd[1 * n + i], bd[2 * n + i], bd[3 * n + i]);
}

__device__ __forceinline__ Command load_command(const FleetBuffers& fb, uint32_t i) {
  const uint32_t n = fb.n;
  return prepare_command(fb.modes[i], fb.targets[0 * n + i], fb.targets[1 * n + i], fb.targets[2 * n + i],
                         fb.targets[3 * n + i]);
}

// What a launch reads of one vehicle, as it is in memory. It is requested
// before anything waits for the command (whose angles go through sincosf, a
// branch that no load moves across): a single-step launch then waits for memory
// once instead of twice.
template <int NROT> struct VehicleRows {
  VState s;
  float u[NROT], body[4];
};
template <int NROT> __device__ __forceinline__ VehicleRows<NROT> load_vehicle(const FleetBuffers& fb, uint32_t env) {
  const uint32_t n = fb.n;
  VehicleRows<NROT> v;
  v.s = load_state(fb.state, n, env);
#pragma unroll
  for (int k = 0; k < NROT; ++k) v.u[k] = fb.motors[k * n + env];
#pragma unroll
  for (int k = 0; k < 4; ++k) v.body[k] = fb.body[k * n + env];
  return v;
}

// Overwrites one environment with its reset draw for `epoch`.
template <int NROT>
__device__ __forceinline__ void reset_in_registers(VState& s, float (&u)[NROT], float m, uint32_t env,
                                                   uint32_t epoch, uint32_t seed_lo, uint32_t seed_hi) {
  ResetValues r = draw_reset(seed_lo, seed_hi, env, epoch);
  s.p = {r.p[0], r.p[1], r.p[2]};
  s.v = {r.v[0], r.v[1], r.v[2]};
  s.q = {r.q[0], r.q[1], r.q[2], r.q[3]};
  s.w = {0.f, 0.f, 0.f};
  float hv = hover_per_motor(m, NROT);
#pragma unroll
  for (int k = 0; k < NROT; ++k) u[k] = hv;
}

// Appends the envs whose predicate is set to the compact list: one ballot and
// one atomicAdd per warp, ranks from __popc of the lower lanes. Every lane of
// the warp must call it.
__device__ __forceinline__ void append_compact(bool pred, uint32_t env, uint32_t* ids, uint32_t* count) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned mask = __ballot_sync(0xFFFFFFFFu, pred);
  if (mask == 0u) return;
  const int leader = __ffs(mask) - 1;
  uint32_t base = 0;
  if ((int)lane == leader) base = atomicAdd(count, (uint32_t)__popc(mask));
  base = __shfl_sync(0xFFFFFFFFu, base, leader);
  if (pred) ids[base + __popc(mask & ((1u << lane) - 1u))] = env;
}

// Box sources of the per-vehicle loop. any_hit(p, r, r2, n_obs, near,
// all, m) says whether the sphere of radius r at p touches a box; m receives a
// squared distance that no box is nearer than (see EnvBoxes). all: every box
// gets the exact test.

// No boxes at all (a fleet without obstacles).
struct NoBoxSource {
  __device__ __forceinline__ NoBoxSource(const FleetBuffers&, uint32_t) {}
  __device__ __forceinline__ bool any_hit(V3, float, float, int, float, bool, float& m) const {
    m = __int_as_float(0x7f800000);
    return false;
  }
};

// The box records of environment env. A test first reads every box's
// circumscribed sphere, one 16-byte load each, and runs the exact test only on
// the boxes whose sphere comes within r + near. A launch's last test needs the
// decision only and takes near = kBoxSlack; the others take kBoxNear, or
// kBoxNearShort in calls of up to kShortCall steps, where a vehicle gets no
// further, so that the clearance is exact up to near and at least the distance
// to the other spheres. 674,653 quads among 10 boxes, a reset and 2 / 6 / 20 / 32 /
// 64 / 256 steps: 144.0 / 185.5 / 288.5 / 374.5 / 601 / 1,978 us with the shorter
// reach throughout, 146.6 / 188.5 / 289.7 / 372.0 / 597 / 1,955 with the longer;
// they meet between 20 and 32 steps. (0.1 and 0.05 m do as 0.2 m does.)
// The sphere's distance is taken low by 3e-4 of the centre distance, which
// covers the hardware square root and a quaternion whose norm is off by the
// 1e-4 that ag_set_obstacles admits, and kBoxSlack covers the rest of the
// rounding, so a box without an exact test is one the exact float32 test
// would have found clear: every decision is the exact test's. Distances that
// are not finite numbers get the exact test.
// A single step over 16 random boxes (centres U[-5, 5]^3, half-extents
// U[0.1, 1]) tests about 0.13 boxes per vehicle exactly, so it reads 16 bytes
// per box and little more instead of 40: a task step of 131,072 environments
// (RK4 x 4) took 37 us a pass instead of 60, and the bench fleet's 1,000-step
// call from fresh states 53.8 ms instead of 57.9 (both less since). There
// kBoxNear hardly matters: 0.25 and 1 m measured 53.9 ms.
constexpr float kBoxSlack = 1e-3f, kBoxNearShort = 0.2f, kBoxNear = 0.5f;  // m
constexpr int kShortCall = 32;

// Boxes that are large and flat gain nothing: every vehicle of a room lies within
// a wall's sphere, so a test reads 64 bytes of a wall instead of 40 and twice the
// instructions. Calls of many steps among nothing but walls (5 x 5 x 0.05 m) take
// longer than with a test of every box from rows in pairs (65,536 quads x 8 walls x
// 200 steps 325 us against 279, x 6 of 16 boxes 382 against 380).
// GROUPED: the spheres are loaded in whole groups (8, or 16 while more than 8
// are left) before any is looked at, so that a group waits for memory once. It
// serves the single-step kernels, where every thread tests (131,072 quads with
// 3 / 8 / 16 / 32 boxes: 23.3 / 27.6 / 34.7 / 52.5 us a pass); in the launches
// of many steps, where few do, the plain loop leaves more registers to the
// step (1M x 1,000 steps: 50.5 ms against 51.6).
// DENSE: while more than two boxes are marked, four are tested at a time (the last
// one again where fewer are left), so that their loads are in flight together. It
// serves the single-step fused kernel and the unfused test; in the task step it
// costs 3 % among 16 small boxes (19.1 -> 19.7 us), and inside the loops of the
// many-step kernel the longer code misses the instruction cache (no_instruction 0.24
// -> 1.15 stalls per issue, 1M x 1,000 steps 10 % slower).
template <bool GROUPED, bool DENSE = false> struct EnvBoxesT {
  const float4* bound;  // this environment's column of box_bound
  const float4* rest;   // and of box_rest
  uint32_t n;
  __device__ __forceinline__ EnvBoxesT(const FleetBuffers& fb, uint32_t env)
      : bound(fb.box_bound + env), rest(fb.box_rest + 2 * (size_t)env), n(fb.n) {}
  __device__ __forceinline__ float dist2(V3 p, int k) const {
    const float4 b = bound[(size_t)k * n], h = rest[2 * (size_t)k * n], q = rest[2 * (size_t)k * n + 1];
    return box_dist2(p, V3{b.x, b.y, b.z}, V3{h.x, h.y, h.z}, Q4{h.w, q.x, q.y, q.z});
  }
  // The distance from p to the sphere b, low by the margin above. The squared
  // centre distance starts from kTiny, far below what the margins see, so the
  // hardware root never gets a zero or a subnormal, which it takes for zero
  // (its infinity would leave out a box around whose centre the vehicle is).
  static __device__ __forceinline__ float low_distance(V3 p, float4 b) {
    constexpr float kTiny = 1e-37f;
    const V3 v = p - V3{b.x, b.y, b.z};
    const float d2 = fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, kTiny)));
    return fmaf(d2 * rsqrt_ftz(d2), 1.f - 3e-4f, -b.w);
  }
  // Spheres k0 .. k0 + G - 1 (the last box again beyond n_obs), bits from bit.
  template <int G>
  __device__ __forceinline__ void scan(V3 p, int k0, int n_obs, int bit, float reach, float& far, uint32_t& exact) const {
    float4 b[G];
#pragma unroll
    for (int j = 0; j < G; ++j) b[j] = bound[(size_t)min(k0 + j, n_obs - 1) * n];
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const float low = low_distance(p, b[j]);
      if (low > reach) far = fminf(far, low);
      else if (k0 + j < n_obs) exact |= 1u << (bit + j);
    }
  }
  __device__ __forceinline__ bool any_hit(V3 p, float r, float r2, int n_obs, float near, bool all, float& m) const {
    const float inf = __int_as_float(0x7f800000);
    const float reach = all ? inf : r + near;
    float far = inf, near2 = inf;  // over the spheres out of reach; over the exact tests (squared)
    bool hit = false;
    for (int k0 = 0; k0 < n_obs; k0 += 32) {
      const int count = min(32, n_obs - k0);
      uint32_t exact = 0;
      if (GROUPED) {
        for (int j = 0; j < count;) {
          if (count - j <= 8) {
            scan<8>(p, k0 + j, n_obs, j, reach, far, exact);
            j += 8;
          } else {
            scan<16>(p, k0 + j, n_obs, j, reach, far, exact);
            j += 16;
          }
        }
      } else {
#pragma unroll 8
        for (int j = 0; j < count; ++j) {
          const float low = low_distance(p, bound[(size_t)(k0 + j) * n]);
          if (low > reach) far = fminf(far, low);
          else exact |= 1u << j;
        }
      }
      while (DENSE && __popc(exact) > 2) {
        float4 b[4], h[4], q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const size_t at = (size_t)(k0 + __ffs(exact) - 1) * n;
          b[i] = bound[at];
          h[i] = rest[2 * at];
          q[i] = rest[2 * at + 1];
          const uint32_t less = exact & (exact - 1);
          exact = i < 3 && less == 0 ? exact : less;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float e2 = box_dist2(p, V3{b[i].x, b[i].y, b[i].z}, V3{h[i].x, h[i].y, h[i].z},
                                     Q4{h[i].w, q[i].x, q[i].y, q[i].z});
          near2 = fminf(near2, e2);
          hit |= touches(r2, e2);
        }
      }
      while (exact) {
        const int j = __ffs(exact) - 1;
        exact &= exact - 1;
        const float e2 = dist2(p, k0 + j);
        near2 = fminf(near2, e2);
        hit |= touches(r2, e2);
      }
    }
    m = fminf(near2, far * far);
    return hit;
  }
};
using EnvBoxes = EnvBoxesT<false>;

// The records of box k of environment env from its ten fields (ag_set_obstacles).
__device__ __forceinline__ void pack_box(const FleetBuffers& fb, uint32_t k, uint32_t env, const float (&v)[10]) {
  const size_t at = (size_t)k * fb.n + env;
  fb.box_bound[at] = make_float4(v[0], v[1], v[2], sqrtf(fmaf(v[5], v[5], fmaf(v[4], v[4], v[3] * v[3]))));
  fb.box_rest[2 * at] = make_float4(v[3], v[4], v[5], v[6]);
  fb.box_rest[2 * at + 1] = make_float4(v[7], v[8], v[9], 0.f);
}

// New poses for every box of environment env, written to its records (the
// half-extents and the sphere radius stay).
static __device__ __noinline__ void redraw_boxes(float4* box_bound, float4* box_rest, const BoxRandDev* box_rand,
                                                 uint32_t n, uint32_t n_obs, uint32_t env, uint32_t epoch,
                                                 uint32_t seed_lo, uint32_t seed_hi) {
  for (uint32_t k = 0; k < n_obs; ++k) {
    float c[3], q[4];
    draw_box_pose(seed_lo, seed_hi, env, epoch, k, box_rand[k], c, q);
    float4* const bound = box_bound + (size_t)k * n + env;
    float4* const rest = box_rest + 2 * ((size_t)k * n + env);
    *bound = make_float4(c[0], c[1], c[2], bound->w);
    rest[0].w = q[0];
    rest[1] = make_float4(q[1], q[2], q[3], 0.f);
  }
}
__device__ __forceinline__ void redraw_boxes(const FleetBuffers& fb, uint32_t env, uint32_t epoch, uint32_t seed_lo,
                                             uint32_t seed_hi) {
  redraw_boxes(fb.box_bound, fb.box_rest, fb.box_rand, fb.n, fb.n_obs, env, epoch, seed_lo, seed_hi);
}

// Resets environment env in device memory (the ag_reset draw): epoch + 1,
// Philox state draw, every motor at hover, zero for the unused ones, and new
// box poses when re-placement is on.
__device__ __forceinline__ void reset_env(const FleetBuffers& fb, uint32_t env, uint32_t seed_lo, uint32_t seed_hi) {
  const uint32_t n = fb.n;
  const uint32_t epoch = fb.epoch[env] + 1u;
  fb.epoch[env] = epoch;
  ResetValues r = draw_reset(seed_lo, seed_hi, env, epoch);
  float* st = fb.state;
  st[0 * n + env] = r.p[0]; st[1 * n + env] = r.p[1]; st[2 * n + env] = r.p[2];
  st[3 * n + env] = r.v[0]; st[4 * n + env] = r.v[1]; st[5 * n + env] = r.v[2];
  st[6 * n + env] = r.q[0]; st[7 * n + env] = r.q[1]; st[8 * n + env] = r.q[2]; st[9 * n + env] = r.q[3];
  st[10 * n + env] = 0.f; st[11 * n + env] = 0.f; st[12 * n + env] = 0.f;
  const int nrot = rotor_count(fb, env);
  const float hv = hover_per_motor(fb.body[env], nrot);
  for (int k = 0; k < 8; ++k) fb.motors[k * n + env] = k < nrot ? hv : 0.f;
  if (fb.box_rand) redraw_boxes(fb, env, epoch, seed_lo, seed_hi);
}

// How far a vehicle may move from p, where a test found no box nearer than
// the squared distance min_e2, before the sphere of radius r could
// touch one; returned squared, or -1 when it must be tested again at once.
// The distance to a box is 1-Lipschitz in the position, so as long as
// |p' - p| < sqrt(min_e2) - r - slack no box is within r of p'. The slack
// (1 mm plus 1e-5 of the magnitudes involved) is far above the float32
// rounding of the test, so a skipped test is one the exact float32 test
// would also have found clear: every collision decision is the exact test's.
__device__ __forceinline__ float clearance_threshold2(V3 p, float min_e2, float r) {
  const float c = sqrtf(min_e2) - r;
  const float slack = 1e-3f + 1e-5f * (fabsf(c) + fabsf(p.x) + fabsf(p.y) + fabsf(p.z));
  const float t = c - slack;
  return t > 0.f ? t * t : -1.f;
}

// When one thread of a warp has to test, the others wait for it anyway: those
// that have moved at least half their clearance (this share of its square)
// test along with it instead of holding the warp up again soon after. Tests
// run early decide what tests run in time would. 1,048,576 quads among 16
// boxes x 1,000 steps: 52.7 -> 50.9 ms (48.5 ms without any test after the
// first step); shares of 0.5, 0.1, 0.03 and 0 measured 51.1, 50.9, 51.0, 51.0.
constexpr float kJoinTest = 0.25f;

// The per-vehicle body of the fused kernels, specialised on the rotor count:
// n_steps steps of `substeps` substeps, then the sphere-vs-box test against
// n_obs boxes and, on a hit, the Philox reset keyed (seed_lo, seed_hi).
// This is simulate() with the command given (cm_in) instead of read from fb; returns
// the final state, which it also stores. MODE >= 0: every calling thread's
// command mode is MODE; the mode is then a constant of the compiled loop,
// and the controller's branches on it fold away.
template <int NROT, int INTEG, bool DRAG, class Boxes, int MODE = -1>
__device__ __forceinline__ VState simulate_cmd(const FleetBuffers& fb, const StepParams& P, uint32_t env,
                                               const VehicleRows<NROT>& rows, const Command& cm_in, int n_steps,
                                               int substeps, int n_obs, const Boxes& boxes, uint32_t seed_lo,
                                               uint32_t seed_hi, uint32_t& resets, bool& any_hit, uint32_t& tests) {
  Command cm = cm_in;
  if (MODE >= 0) cm.mode = MODE;
  const uint32_t n = fb.n;
  VState s = rows.s;
  normalize(s.q);
  float u[NROT];
#pragma unroll
  for (int k = 0; k < NROT; ++k) u[k] = rows.u[k];
  const Body b = make_body(rows.body[0], rows.body[1], rows.body[2], rows.body[3]);
  // Collision tests that cannot hit are skipped (see clearance_threshold2):
  // p_test is the position of the last test, thr2 the squared distance
  // the vehicle may move from there before it could touch a box (-1: test
  // at the next step).
  V3 p_test = {0.f, 0.f, 0.f};
  float thr2 = -1.f;
  const float r = sqrtf(P.r2);
  const unsigned group = __activemask();  // threads of one launch, so of one trip count
  for (int step = 0; step < n_steps; ++step) {
    for (int ss = 0; ss < substeps; ++ss) {
      V3 b3;
      Wrench4 W = allocate<NROT>(controller(s, cm, b, P, b3), u, P);
      integrate<INTEG, DRAG>(s, b3, W, b, P);
    }
    if (n_obs > 0) {
      const V3 dp = s.p - p_test;
      const float moved2 = dot(dp, dp);
      if (n_steps == 1 || (__any_sync(group, !(moved2 < thr2)) && !(moved2 < kJoinTest * thr2))) {
        float min_e2;
        const bool hit = boxes.any_hit(s.p, r, P.r2, n_obs, step + 1 == n_steps ? kBoxSlack : n_steps <= kShortCall ? kBoxNearShort : kBoxNear,
                                       P.exact_tests != 0, min_e2);
        tests += 1;
        p_test = s.p;
        thr2 = P.exact_tests ? -1.f : clearance_threshold2(s.p, min_e2, r);
        if (hit) {
          any_hit = true;
          resets += 1;
          const uint32_t epoch = fb.epoch[env] + 1u;  // read and written only where a reset needs it
          fb.epoch[env] = epoch;
          reset_in_registers<NROT>(s, u, b.m, env, epoch, seed_lo, seed_hi);
          thr2 = -1.f;
          if (fb.box_rand) redraw_boxes(fb, env, epoch, seed_lo, seed_hi);
        }
      }
    }
  }
  store_state(fb.state, n, env, s);
#pragma unroll
  for (int k = 0; k < NROT; ++k) fb.motors[k * n + env] = u[k];
  return s;
}

// With BY_MODE and the grouped thread order (fb.order: warps of one rotor
// count and command mode), a group of threads that run together and share
// one command mode (position, body velocity, attitude + thrust) runs the
// steps compiled for that mode, in which the controller's branches on the
// mode are folded away; other threads run the branching form. Every fused
// multiply-add of the step is explicit (fmaf) and the files that include
// this header are compiled without contraction, so both forms round
// identically and the choice changes no result.
template <int NROT, int INTEG, bool DRAG, bool BY_MODE = false, class Boxes>
__device__ __forceinline__ void simulate(const FleetBuffers& fb, const StepParams& P, uint32_t env,
                                         int n_steps, int substeps, int n_obs, const Boxes& boxes, uint32_t seed_lo,
                                         uint32_t seed_hi, uint32_t& resets, bool& any_hit, uint32_t& tests) {
  const VehicleRows<NROT> rows = load_vehicle<NROT>(fb, env);
  const Command cm = load_command(fb, env);
  bool uniform = false;
  if (BY_MODE && fb.order) {
    const unsigned group = __activemask();
    uniform = __match_any_sync(group, cm.mode) == group;
  }
  if (uniform) {
    if (cm.mode == kModePosition) {
      simulate_cmd<NROT, INTEG, DRAG, Boxes, kModePosition>(fb, P, env, rows, cm, n_steps, substeps, n_obs, boxes,
                                                           seed_lo, seed_hi, resets, any_hit, tests);
      return;
    }
    if (cm.mode == kModeBodyVel) {
      simulate_cmd<NROT, INTEG, DRAG, Boxes, kModeBodyVel>(fb, P, env, rows, cm, n_steps, substeps, n_obs, boxes,
                                                          seed_lo, seed_hi, resets, any_hit, tests);
      return;
    }
    if (cm.mode == kModeAttThrust) {
      simulate_cmd<NROT, INTEG, DRAG, Boxes, kModeAttThrust>(fb, P, env, rows, cm, n_steps, substeps, n_obs, boxes,
                                                            seed_lo, seed_hi, resets, any_hit, tests);
      return;
    }
  }
  simulate_cmd<NROT, INTEG, DRAG>(fb, P, env, rows, cm, n_steps, substeps, n_obs, boxes, seed_lo, seed_hi, resets,
                                  any_hit, tests);
}

}  // namespace agk
