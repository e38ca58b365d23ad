// adjoint.cu — differentiable rollout: recorded forward + hand-written adjoint.
//
// Objective (per environment i, over a recorded rollout of H steps):
//   L_i = sum_{t=1..H} ( w_pos |p_t - p_goal,i|^2 + w_omega |Omega_t|^2 ),
// with x_t the state after step t. Gradients are taken with respect to the
// initial state x_0 (13 numbers per environment), the 12 diagonal controller
// gains (k_x, k_v, k_R, k_Omega), shared by the fleet, and each environment's
// four command targets.
//
// The differentiated step is the controller of the environment's command mode
// (position tracking, Sec. I after Lee et al. 2011; body velocity, Eqs. 6-9;
// attitude and thrust, Eqs. 1-2; or a direct wrench) with the attitude law
// of Sec. IV-A (Eqs. 3-5), rotor allocation with per-motor clamp (subgradient
// 0 on a clamped motor) and first-order lag, and the semi-implicit Euler
// update with quaternion renormalisation. Reverse mode is written out by hand;
// the comments name the forward line each block inverts.
//
// What is recorded. A step's reverse needs its start state (13 floats), the
// realised thrust W.f and which motors passed the clamp (one bit each): 15
// words, kept as four float4 per vehicle and step (64 bytes), so the record
// stores and the sweep loads four 16-byte words per step and nothing of the
// allocation, the lag or the integration is computed again. The end state of
// a step is the next entry's start state. The record writes every entry as
// it goes when a tape of the whole horizon fits (AdjointBuffers::full_tape);
// otherwise it keeps a checkpoint (state + motors) every K steps and the sweep
// recomputes one segment's entries at a time.
//
// Thread slot s handles environment order[s] (grouped by rotor type and
// command mode, as in the fused step): a warp runs one mode's code. The tape and
// the norm of q_0 are kept in slot order, so their rows are read and written
// coalesced whatever the modes are. Checkpoints are kept by environment: they
// grow with the horizon, and the padding slots of a fleet of one would make them
// 96 times as large.
//
// Attitude adjoint. The adjoint of the unit quaternion is carried as the
// 3-vector g of the right perturbation q -> q (1, delta / 2): the step's
// q' = q c / |c|, c = (1, h/2 Omega'), turns it by R(c), and every use of
// R = R(q) adds a short body-frame vector to it. That replaces the adjoints
// of q (4), of R's nine entries and of the normalisation.
//
// The file is compiled without implicit contraction and every fused
// multiply-add is explicit, so the record rounds alike in both forms.
#include <cstdint>
#include <cuda_runtime.h>

#include "adjoint_internal.h"
#include "fleet_device.cuh"

namespace agk {
namespace {

// One vehicle during the forward rollout.
template <int NROT> struct Vehicle {
  VState s;
  float u[NROT];
};

// ------------------------------------------------------------------- tape --
// Entry of a step: (p, v.x) (v.y, v.z, Omega.x, Omega.y) (q) (Omega.z, W.f, pass bits, 0).
struct TapeStep {
  V3 p, v;
  Q4 q;
  V3 w;
  float wf;
  uint32_t pass;
};

__device__ __forceinline__ void store_entry(float4* __restrict__ e, size_t n, const VState& s, float wf, uint32_t pass) {
  e[0] = make_float4(s.p.x, s.p.y, s.p.z, s.v.x);
  e[n] = make_float4(s.v.y, s.v.z, s.w.x, s.w.y);
  e[2 * n] = make_float4(s.q.w, s.q.x, s.q.y, s.q.z);
  e[3 * n] = make_float4(s.w.z, wf, __uint_as_float(pass), 0.f);
}

__device__ __forceinline__ TapeStep unpack(float4 a, float4 b, float4 c, float4 d) {
  return {{a.x, a.y, a.z}, {a.w, b.x, b.y}, {c.x, c.y, c.z, c.w}, {b.z, b.w, d.x}, d.y, __float_as_uint(d.z)};
}

// ---------------------------------------------------------------- forward --
// One recorded step from s (unit quaternion): controller -> allocation, clamp
// and lag -> semi-implicit Euler, the fused step's own functions.
template <int NROT, int MODE>
__device__ __forceinline__ void forward_step(Vehicle<NROT>& x, const Command& cm, const Body& b, const StepParams& P,
                                             float& wf, uint32_t& pass) {
  V3 b3;
  const Wrench4 cmd = controller(x.s, cm, b, P, b3);
  const Wrench4 W = allocate<NROT>(cmd, x.u, P, &pass);
  wf = W.f;
  step_sie<true>(x.s, b3, W, b, P.drag, P.h);
}

template <int NROT>
__device__ __forceinline__ void load_vehicle(const float* st, const float* mot, uint32_t n, uint32_t i, Vehicle<NROT>& x) {
  x.s.p = {st[0 * n + i], st[1 * n + i], st[2 * n + i]};
  x.s.v = {st[3 * n + i], st[4 * n + i], st[5 * n + i]};
  x.s.q = {st[6 * n + i], st[7 * n + i], st[8 * n + i], st[9 * n + i]};
  x.s.w = {st[10 * n + i], st[11 * n + i], st[12 * n + i]};
#pragma unroll
  for (int k = 0; k < NROT; ++k) x.u[k] = mot[k * n + i];
}

template <int NROT>
__device__ __forceinline__ void store_vehicle(float* st, float* mot, uint32_t n, uint32_t i, const Vehicle<NROT>& x) {
  const VState& s = x.s;
  st[0 * n + i] = s.p.x; st[1 * n + i] = s.p.y; st[2 * n + i] = s.p.z;
  st[3 * n + i] = s.v.x; st[4 * n + i] = s.v.y; st[5 * n + i] = s.v.z;
  st[6 * n + i] = s.q.w; st[7 * n + i] = s.q.x; st[8 * n + i] = s.q.y; st[9 * n + i] = s.q.z;
  st[10 * n + i] = s.w.x; st[11 * n + i] = s.w.y; st[12 * n + i] = s.w.z;
#pragma unroll
  for (int k = 0; k < NROT; ++k) mot[k * n + i] = x.u[k];
}

__device__ __forceinline__ Body body_at(const AdjointBuffers& ab, uint32_t i) {
  const uint32_t n = ab.n;
  return make_body(ab.body[i], ab.body[n + i], ab.body[2 * n + i], ab.body[3 * n + i]);
}

__device__ __forceinline__ int rotors_of(const AdjointBuffers& ab, uint32_t i) {
  return i < ab.n_quad ? 4 : (i < ab.n_quad + ab.n_hexa ? 6 : 8);
}

template <int MODE> __device__ __forceinline__ Command command_at(const AdjointBuffers& ab, uint32_t i) {
  const uint32_t n = ab.n;
  Command cm = prepare_command(MODE, ab.targets[i], ab.targets[n + i], ab.targets[2 * n + i], ab.targets[3 * n + i]);
  cm.mode = MODE;
  return cm;
}

__device__ __forceinline__ int mode_of(const AdjointBuffers& ab, uint32_t i) {
  const int m = ab.modes[i];
  return m > kModeWrench ? kModeWrench : m;
}

// Calls f.template run<NROT, MODE>() for environment i's airframe and mode.
template <int NROT, class F> __device__ __forceinline__ void by_mode(int mode, const F& f) {
  switch (mode) {
    case kModePosition: f.template run<NROT, kModePosition>(); break;
    case kModeBodyVel: f.template run<NROT, kModeBodyVel>(); break;
    case kModeAttThrust: f.template run<NROT, kModeAttThrust>(); break;
    default: f.template run<NROT, kModeWrench>(); break;
  }
}
template <class F> __device__ __forceinline__ void by_airframe_and_mode(int rotors, int mode, const F& f) {
  if (rotors == 4) by_mode<4>(mode, f);
  else if (rotors == 6) by_mode<6>(mode, f);
  else by_mode<8>(mode, f);
}

// Forward recording of slot's environment: n_steps steps from the fleet state,
// tape entries (FULL_TAPE) or checkpoints every K steps, loss, final state,
// saturation flag.
template <bool FULL_TAPE> struct Record {
  const AdjointBuffers& ab;
  const StepParams& P;
  uint32_t slot, env;
  template <int NROT, int MODE> __device__ __forceinline__ void run() const {
    const uint32_t n = ab.n, ns = ab.n_slots;
    Vehicle<NROT> x;
    load_vehicle(ab.state, ab.motors, n, env, x);
    ab.inv_q0[slot] = 1.f / sqrtf(dot4(x.s.q));
    normalize(x.s.q);
    const Body b = body_at(ab, env);
    const Command cm = command_at<MODE>(ab, env);
    const V3 goal = {ab.goal_in[env], ab.goal_in[n + env], ab.goal_in[2 * n + env]};
    ab.p_goal[env] = goal.x;
    ab.p_goal[n + env] = goal.y;
    ab.p_goal[2 * n + env] = goal.z;
    float loss = 0.f;
    uint32_t all_pass = (1u << NROT) - 1u;
    float4* entry = ab.tape + slot;
    float* ckpt = ab.ckpt;
    int to_ckpt = 0;
    for (int t = 0; t < ab.n_steps; ++t) {
      if (!FULL_TAPE && to_ckpt-- == 0) {
        store_vehicle(ckpt, ckpt + 13 * (size_t)n, n, env, x);
        ckpt += 21 * (size_t)n;
        to_ckpt = ab.K - 1;
      }
      const VState start = x.s;
      float wf;
      uint32_t pass = 0;
      forward_step<NROT, MODE>(x, cm, b, P, wf, pass);
      all_pass &= pass;
      if (FULL_TAPE) {
        store_entry(entry, ns, start, wf, pass);
        entry += 4 * (size_t)ns;
      }
      const V3 e = x.s.p - goal;
      loss += fmaf(ab.w_omega, dot(x.s.w, x.s.w), ab.w_pos * dot(e, e));
    }
    if (FULL_TAPE) store_entry(entry, ns, x.s, 0.f, 0u);  // entry H: the end state
    store_vehicle(ab.state, ab.motors, n, env, x);
    ab.loss[env] = loss;
    ab.saturated[env] = all_pass == (1u << NROT) - 1u ? 0 : 1;
  }
};

// One warp per block: the fleet's warps spread evenly over the SMs (a
// 65,536-vehicle fleet puts 13 or 14 on each of 152 SMs, where 128-thread
// blocks would put 12 on some and 16 on others). Writing the tape here costs
// little beside the step: 65,536 quads x 256 steps take 193 us at 5.6 TB/s of
// tape, against 176 us without it and another 194 us to recompute it later.
constexpr int kRecordBlock = 32;
template <bool FULL_TAPE>
__global__ void __launch_bounds__(kRecordBlock) k_record(AdjointBuffers ab, StepParams P) {
  const uint32_t slot = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t env = ab.order[slot];  // n_slots is a multiple of the block
  if (env >= ab.n) return;
  by_airframe_and_mode(rotors_of(ab, env), mode_of(ab, env), Record<FULL_TAPE>{ab, P, slot, env});
}

// ---------------------------------------------------------------- backward --
// Adjoint state of one vehicle during the reverse sweep: of the state after a
// step (g: the attitude's right perturbation), of the gains and the targets.
template <int NROT> struct Adj {
  V3 p, v, g, w;
  float u[NROT];
};
struct ParamAdj {
  V3 kx, kv, kR, kW;
  float tb[4];
};

__device__ __forceinline__ V3 mul3(V3 a, V3 b) { return {a.x * b.x, a.y * b.y, a.z * b.z}; }
__device__ __forceinline__ V3 fma3(float s, V3 a, V3 c) { return {fmaf(s, a.x, c.x), fmaf(s, a.y, c.y), fmaf(s, a.z, c.z)}; }
__device__ __forceinline__ V3 fma33(V3 a, V3 b, V3 c) { return {fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y), fmaf(a.z, b.z, c.z)}; }
__device__ __forceinline__ V3 neg3(V3 a) { return {-a.x, -a.y, -a.z}; }
// c + a x b
__device__ __forceinline__ V3 cross_add(V3 a, V3 b, V3 c) {
  return {fmaf(a.y, b.z, fmaf(-a.z, b.y, c.x)), fmaf(a.z, b.x, fmaf(-a.x, b.z, c.y)), fmaf(a.x, b.y, fmaf(-a.y, b.x, c.z))};
}
// c + x_bar of y = x / |x| (1 / |x| = in): in (y_bar - y (y . y_bar))
__device__ __forceinline__ V3 normalize_bwd_add(V3 y, float in, V3 ybar, V3 c) {
  const float d = dot(y, ybar);
  return fma3(in, fma3(-d, y, ybar), c);
}

// Reverse of forward_step from its tape entry x and the position and body
// rate after it. On entry z is the adjoint of (x_{t+1}, u_{t+1}) without this
// step's loss term, on exit that of (x_t, u_t). cp2 and cw2 are 2 w_pos and
// 2 w_omega times the environment's loss weight.
template <int NROT, int MODE>
__device__ __forceinline__ void backward_step(const TapeStep& x, V3 pn, V3 wn, const Command& cm, const Body& b,
                                              const StepParams& P, V3 goal, float cp2, float cw2, Adj<NROT>& z,
                                              ParamAdj& gb) {
  constexpr int T = NROT == 4 ? 0 : (NROT == 6 ? 1 : 2);
  const float h = P.h;
  // the loss term of x_{t+1}
  const V3 pb = fma3(cp2, pn - goal, z.p);
  V3 wb = fma3(cw2, wn, z.w);
  // q' = q (1, hw) / s with hw = h/2 Omega', s^2 = 1 + |hw|^2:
  // Omega'_bar += h / s^2 (g + hw x g), g <- R(c) g = g + 2 / s^2 (hw x g + hw x (hw x g))
  const V3 hw = (0.5f * h) * wn;
  const float is2 = rcp_ftz(fmaf(hw.z, hw.z, fmaf(hw.y, hw.y, fmaf(hw.x, hw.x, 1.f))));
  const V3 t1 = cross(hw, z.g);
  wb = fma3(h * is2, z.g + t1, wb);  // now the adjoint of Omega' (and of Omega through Omega' = Omega + ...)
  V3 g = fma3(2.f * is2, cross_add(hw, t1, t1), z.g);
  // p' = p + h v';  v' = v + h (W.f/m b3 - (c/m) v + g e3)
  const V3 vnb = fma3(h, pb, z.v);
  const float him = h * b.inv_m;
  V3 vb = fmaf(-him, P.drag, 1.f) * vnb;
  float R[3][3];
  rotation(x.q, R);
  const V3 r0 = {R[0][0], R[1][0], R[2][0]}, r1 = {R[0][1], R[1][1], R[2][1]}, r2 = {R[0][2], R[1][2], R[2][2]};
  const float Wfb = him * dot(r2, vnb);
  V3 tilt = (him * x.wf) * vnb;  // world adjoint of b3: g gets e3 x (R^T tilt) once all its terms are in
  // Omega' = Omega + h J^-1 (W.M - gyro)
  const V3 wmb = {(h * b.ijx) * wb.x, (h * b.ijy) * wb.y, (h * b.ijz) * wb.z};
  // u' = u + alpha (clamp(A^+ (f, M)) - u), W = A u': motors as FP32 pairs, the commanded wrench's adjoint as
  // (f, M_x) and (M_y, M_z)
  float2 Ma = make_float2(0.f, 0.f), Mc = make_float2(0.f, 0.f);
  {
    const float2 f2 = make_float2(Wfb, Wfb), x2 = make_float2(wmb.x, wmb.x), y2 = make_float2(wmb.y, wmb.y),
                 z2 = make_float2(wmb.z, wmb.z), keep2 = make_float2(1.f - P.alpha, 1.f - P.alpha),
                 al2 = make_float2(P.alpha, P.alpha);
#pragma unroll
    for (int j = 0; j < NROT / 2; ++j) {
      const int i = 2 * j;
      float2 un = make_float2(z.u[i], z.u[i + 1]);
      un = __ffma2_rn(make_float2(P.A[T][0][i], P.A[T][0][i + 1]), f2, un);
      un = __ffma2_rn(make_float2(P.A[T][1][i], P.A[T][1][i + 1]), x2, un);
      un = __ffma2_rn(make_float2(P.A[T][2][i], P.A[T][2][i + 1]), y2, un);
      un = __ffma2_rn(make_float2(P.A[T][3][i], P.A[T][3][i + 1]), z2, un);
      const float2 k = __fmul2_rn(keep2, un);
      z.u[i] = k.x;
      z.u[i + 1] = k.y;
      float2 c = __fmul2_rn(al2, un);
      c.x = (x.pass >> i) & 1u ? c.x : 0.f;
      c.y = (x.pass >> (i + 1)) & 1u ? c.y : 0.f;
      const float2 cx = make_float2(c.x, c.x), cy = make_float2(c.y, c.y);
      Ma = __ffma2_rn(make_float2(P.Ap[T][i][0], P.Ap[T][i][1]), cx, Ma);
      Mc = __ffma2_rn(make_float2(P.Ap[T][i][2], P.Ap[T][i][3]), cx, Mc);
      Ma = __ffma2_rn(make_float2(P.Ap[T][i + 1][0], P.Ap[T][i + 1][1]), cy, Ma);
      Mc = __ffma2_rn(make_float2(P.Ap[T][i + 1][2], P.Ap[T][i + 1][3]), cy, Mc);
    }
  }
  const float Mf = Ma.x;
  const V3 Mm = {Ma.y, Mc.x, Mc.y};
  V3 gyrob = neg3(wmb);
  z.p = pb;
  if (MODE == kModeWrench) {
    gb.tb[0] += Mf; gb.tb[1] += Mm.x; gb.tb[2] += Mm.y; gb.tb[3] += Mm.z;
  } else {
    const V3 kx = {P.kx[0], P.kx[1], P.kx[2]}, kv = {P.kv[0], P.kv[1], P.kv[2]};
    // the step's R_d, commanded yaw rate and their intermediates, as controller() forms them
    V3 rd0, rd1, rd2, a, ex, B0, B1, B2, vV;
    float ian = 0.f, icn = 0.f, irxz = 0.f, rate = 0.f, hc = 1.f, hs = 0.f, cps = 1.f, sps = 0.f, ir = 0.f;
    bool turned = false;
    if (MODE == kModePosition) {
      ex = {x.p.x - cm.c[0], x.p.y - cm.c[1], x.p.z - cm.c[2]};
      a = {fmaf(-kx.x, ex.x, -(kv.x * x.v.x)), fmaf(-kx.y, ex.y, -(kv.y * x.v.y)),
           fmaf(-kx.z, ex.z, fmaf(-kv.z, x.v.z, kGravity))};
      const float a2 = dot(a, a);
      ian = a2 > 1e-18f ? rsqrt_ftz(a2) : 0.f;
      rd2 = ian > 0.f ? ian * a : V3{0.f, 0.f, 1.f};
      hc = cm.c[3];
      hs = cm.c[4];
      V3 c = cross_xy(rd2, hc, hs);
      float c2 = dot(c, c);
      turned = !(c2 > 1e-18f);
      if (turned) {
        hc = -cm.c[4];
        hs = cm.c[3];
        c = cross_xy(rd2, hc, hs);
        c2 = dot(c, c);
      }
      icn = rsqrt_ftz(c2);
      rd1 = icn * c;
      rd0 = cross(rd1, rd2);
    } else {
      const float rho2 = fmaf(r0.y, r0.y, r0.x * r0.x);
      if (rho2 >= kMinNormal) {
        ir = rsqrt_ftz(rho2);
        cps = r0.x * ir;
        sps = r0.y * ir;
      }
      float cphi, sphi, cth, sth;
      if (MODE == kModeBodyVel) {
        vV = {fmaf(sps, x.v.y, cps * x.v.x), fmaf(cps, x.v.y, -(sps * x.v.x)), x.v.z};
        a = {kv.x * (cm.c[0] - vV.x), kv.y * (cm.c[1] - vV.y), fmaf(kv.z, cm.c[2] - vV.z, kGravity)};
        const float rxz2 = fmaf(a.z, a.z, a.x * a.x);
        const float an2 = fmaf(a.y, a.y, rxz2);
        cphi = 1.f; sphi = 0.f; cth = 1.f; sth = 0.f;
        if (rxz2 >= kMinNormal) {
          irxz = rsqrt_ftz(rxz2);
          ian = rsqrt_ftz(an2);
          cth = a.z * irxz;
          sth = a.x * irxz;
          cphi = rxz2 * irxz * ian;
          sphi = -a.y * ian;
        } else if (an2 > 0.f) {
          cphi = 0.f;
          sphi = a.y > 0.f ? -1.f : 1.f;
        }
        rate = cm.c[3];
      } else {
        cphi = cm.c[0]; sphi = cm.c[1]; cth = cm.c[2]; sth = cm.c[3]; rate = cm.c[4];
      }
      // columns of R_y(theta_d) R_x(phi_d), then R_d = R_psi times them
      B0 = {cth, 0.f, -sth};
      B1 = {sth * sphi, cphi, cth * sphi};
      B2 = {sth * cphi, -sphi, cth * cphi};
      rd0 = {cps * B0.x, sps * B0.x, B0.z};
      rd1 = {fmaf(cps, B1.x, -(sps * B1.y)), fmaf(sps, B1.x, cps * B1.y), B1.z};
      rd2 = {fmaf(cps, B2.x, -(sps * B2.y)), fmaf(sps, B2.x, cps * B2.y), B2.z};
    }
    // M = -k_R e_R - k_W e_W + gyro(Omega), e_W = Omega - rate R^T e3, 2 e_R = vee(E - E^T), E = R_d^T R
    gyrob = gyrob + Mm;
    const V3 eWb = {-P.kW[0] * Mm.x, -P.kW[1] * Mm.y, -P.kW[2] * Mm.z};
    const V3 eb = {-0.5f * P.kR[0] * Mm.x, -0.5f * P.kR[1] * Mm.y, -0.5f * P.kR[2] * Mm.z};  // of 2 e_R
    const float E00 = dot(rd0, r0), E01 = dot(rd0, r1), E02 = dot(rd0, r2);
    const float E10 = dot(rd1, r0), E11 = dot(rd1, r1), E12 = dot(rd1, r2);
    const float E20 = dot(rd2, r0), E21 = dot(rd2, r1), E22 = dot(rd2, r2);
    const V3 hm = 0.5f * Mm;
    gb.kR = {fmaf(E12 - E21, hm.x, gb.kR.x), fmaf(E20 - E02, hm.y, gb.kR.y), fmaf(E01 - E10, hm.z, gb.kR.z)};
    V3 eW = x.w;
    if (MODE != kModePosition) eW = {fmaf(-rate, R[2][0], x.w.x), fmaf(-rate, R[2][1], x.w.y), fmaf(-rate, R[2][2], x.w.z)};
    gb.kW = {fmaf(-eW.x, Mm.x, gb.kW.x), fmaf(-eW.y, Mm.y, gb.kW.y), fmaf(-eW.z, Mm.z, gb.kW.z)};
    wb = wb + eWb;
    // g += (tr(E) I - E) eb
    g.x = fmaf(E11 + E22, eb.x, fmaf(-E01, eb.y, fmaf(-E02, eb.z, g.x)));
    g.y = fmaf(E00 + E22, eb.y, fmaf(-E10, eb.x, fmaf(-E12, eb.z, g.y)));
    g.z = fmaf(E00 + E11, eb.z, fmaf(-E20, eb.x, fmaf(-E21, eb.y, g.z)));
    // columns of R_d: r_j with the adjoints of E_ij - E_ji
    V3 rd0b = fma3(eb.y, r2, (-eb.z) * r1), rd1b = fma3(eb.z, r0, (-eb.x) * r2), rd2b = fma3(eb.x, r1, (-eb.y) * r0);
    const float mf = b.m * Mf;
    if (MODE == kModePosition) {
      // f = m a . b3
      V3 ab = mf * r2;
      tilt = fma3(mf, a, tilt);
      // b1d = b2d x b3d;  b2d = c / |c|, c = b3d x b1c;  b3d = a / |a| (constant e3 where |a| = 0)
      rd1b = cross_add(rd2, rd0b, rd1b);
      rd2b = cross_add(rd0b, rd1, rd2b);
      const float d = dot(rd1, rd1b);
      const V3 cb = icn * fma3(-d, rd1, rd1b);
      rd2b = {fmaf(hs, cb.z, rd2b.x), fmaf(-hc, cb.z, rd2b.y), fmaf(hc, cb.y, fmaf(-hs, cb.x, rd2b.z))};
      const float hcb = fmaf(cb.y, rd2.z, -(cb.z * rd2.y)), hsb = fmaf(cb.z, rd2.x, -(cb.x * rd2.z));
      if (ian > 0.f) ab = normalize_bwd_add(rd2, ian, rd2b, ab);
      // a = -k_x (p - p_d) - k_v v + g e3
      const V3 xa = mul3(kx, ab);
      z.p = z.p - xa;
      vb = fma33(neg3(kv), ab, vb);
      gb.kx = fma33(neg3(ex), ab, gb.kx);
      gb.kv = fma33(neg3(x.v), ab, gb.kv);
      gb.tb[0] += xa.x;
      gb.tb[1] += xa.y;
      gb.tb[2] += xa.z;
      // b1c = (cos psi_d, sin psi_d, 0), turned by 90 degrees in the fallback: d b1c / d psi_d = (-hs, hc, 0) in both
      gb.tb[3] = fmaf(-hs, hcb, fmaf(hc, hsb, gb.tb[3]));
    } else {
      // e_W's third row of R: g -= rate (eWb x R^T e3)
      const V3 row = {R[2][0], R[2][1], R[2][2]};
      const float rateb = -dot(row, eWb);
      g = cross_add(rate * row, eWb, g);
      // R_d = R_psi B: adjoints of B's columns and of (cos psi, sin psi)
      const V3 B0b = {fmaf(sps, rd0b.y, cps * rd0b.x), fmaf(cps, rd0b.y, -(sps * rd0b.x)), rd0b.z};
      const V3 B1b = {fmaf(sps, rd1b.y, cps * rd1b.x), fmaf(cps, rd1b.y, -(sps * rd1b.x)), rd1b.z};
      const V3 B2b = {fmaf(sps, rd2b.y, cps * rd2b.x), fmaf(cps, rd2b.y, -(sps * rd2b.x)), rd2b.z};
      float cpb = fmaf(rd2b.y, B2.y, fmaf(rd2b.x, B2.x, fmaf(rd1b.y, B1.y, fmaf(rd1b.x, B1.x, rd0b.x * B0.x))));
      float spb = fmaf(rd2b.y, B2.x, fmaf(-rd2b.x, B2.y, fmaf(rd1b.y, B1.x, fmaf(-rd1b.x, B1.y, rd0b.y * B0.x))));
      if (MODE == kModeAttThrust) {
        // B = R_y(theta_d) R_x(phi_d): columns (ct, 0, -st), (st sp, cp, ct sp), (st cp, -sp, ct cp)
        const float cp = cm.c[0], sp = cm.c[1], ct = cm.c[2], st = cm.c[3];
        const float u1 = fmaf(ct, B1b.x, -(st * B1b.z)), u2 = fmaf(ct, B2b.x, -(st * B2b.z));
        const float v1 = fmaf(st, B1b.x, ct * B1b.z), v2 = fmaf(st, B2b.x, ct * B2b.z);
        gb.tb[1] += fmaf(-st, B0b.x, fmaf(-ct, B0b.z, fmaf(sp, u1, cp * u2)));
        gb.tb[0] += fmaf(cp, v1 - B2b.y, -(sp * (v2 + B1b.y)));
        gb.tb[2] += rateb;
        gb.tb[3] += Mf;
      } else {
        // f = m a . (R_psi^T b3)
        const V3 b3V = {fmaf(sps, r2.y, cps * r2.x), fmaf(cps, r2.y, -(sps * r2.x)), r2.z};
        V3 ab = mf * b3V;
        const V3 fb = mf * a;
        tilt = {tilt.x + fmaf(cps, fb.x, -(sps * fb.y)), tilt.y + fmaf(sps, fb.x, cps * fb.y), tilt.z + fb.z};
        cpb = fmaf(r2.x, fb.x, fmaf(r2.y, fb.y, cpb));
        spb = fmaf(r2.y, fb.x, fmaf(-r2.x, fb.y, spb));
        // B from a: B2 = a / |a|, B0 = (a_z, 0, -a_x) / |(a_x, a_z)|, B1 = B2 x B0 (constant when a_x = a_z = 0)
        if (irxz > 0.f) {
          const V3 B2c = cross_add(B0, B1b, B2b), B0c = cross_add(B1b, B2, B0b);
          const float d = fmaf(B0.z, B0c.z, B0.x * B0c.x);
          ab.z = fmaf(irxz, fmaf(-d, B0.x, B0c.x), ab.z);
          ab.x = fmaf(-irxz, fmaf(-d, B0.z, B0c.z), ab.x);
          ab = normalize_bwd_add(B2, ian, B2c, ab);
        }
        // a = k_v (v_d - v^V) + g e3,  v^V = R_psi^T v
        const V3 tv = mul3(kv, ab);
        gb.tb[0] += tv.x;
        gb.tb[1] += tv.y;
        gb.tb[2] += tv.z;
        gb.tb[3] += rateb;
        gb.kv = fma33(V3{cm.c[0] - vV.x, cm.c[1] - vV.y, cm.c[2] - vV.z}, ab, gb.kv);
        vb = {vb.x - fmaf(cps, tv.x, -(sps * tv.y)), vb.y - fmaf(sps, tv.x, cps * tv.y), vb.z - tv.z};
        cpb = fmaf(-x.v.x, tv.x, fmaf(-x.v.y, tv.y, cpb));
        spb = fmaf(-x.v.y, tv.x, fmaf(x.v.x, tv.y, spb));
      }
      // (cos psi, sin psi) = (R00, R10) / |(R00, R10)|; ir = 0 where R00 = R10 = 0
      const float d = fmaf(sps, spb, cps * cpb);
      const float c0 = ir * fmaf(-d, cps, cpb), c1 = ir * fmaf(-d, sps, spb);  // adjoint of (R00, R10)
      g.y = fmaf(-r2.x, c0, fmaf(-r2.y, c1, g.y));
      g.z = fmaf(r1.x, c0, fmaf(r1.y, c1, g.z));
    }
  }
  // b3 = R e3: g += e3 x (R^T tilt)
  g.x -= dot(r1, tilt);
  g.y += dot(r0, tilt);
  // gyro = (gx wy wz, gy wz wx, gz wx wy)
  const V3 gg = {b.gx * gyrob.x, b.gy * gyrob.y, b.gz * gyrob.z};
  z.w = {fmaf(gg.y, x.w.z, fmaf(gg.z, x.w.y, wb.x)), fmaf(gg.x, x.w.z, fmaf(gg.z, x.w.x, wb.y)),
         fmaf(gg.x, x.w.y, fmaf(gg.y, x.w.x, wb.z))};
  z.v = vb;
  z.g = g;
}

// Tape entries in flight per vehicle: the sweep's loads run this many steps
// ahead of their use, asynchronously into shared memory (each thread copies
// and reads its own column, so there is nothing to synchronise between threads).
constexpr int kSweepStages = 4;
constexpr int kAdjointBlock = 32;

__device__ __forceinline__ void copy16_async(float4* dst_shared, const float4* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst_shared);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// Reverse sweep of slot's environment; the gain adjoints are returned in gb.
template <bool FULL_TAPE> struct Sweep {
  const AdjointBuffers& ab;
  const StepParams& P;
  uint32_t slot, env;
  float4 (*ring)[4][kAdjointBlock];  // [kSweepStages][4][lane]
  V3 (&gains)[4];
  template <int NROT, int MODE> __device__ __forceinline__ void run() const {
    const size_t n = ab.n, ns = ab.n_slots;
    const uint32_t lane = threadIdx.x;
    const Body b = body_at(ab, env);
    const Command cm = command_at<MODE>(ab, env);
    const V3 goal = {ab.p_goal[env], ab.p_goal[n + env], ab.p_goal[2 * n + env]};
    const float wgt = ab.loss_weights ? ab.loss_weights[env] : 1.f;
    const float cp2 = 2.f * ab.w_pos * wgt, cw2 = 2.f * ab.w_omega * wgt;
    Adj<NROT> z;
    z.p = z.v = z.g = z.w = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < NROT; ++k) z.u[k] = 0.f;
    ParamAdj gb;
    gb.kx = gb.kv = gb.kR = gb.kW = {0.f, 0.f, 0.f};
    gb.tb[0] = gb.tb[1] = gb.tb[2] = gb.tb[3] = 0.f;
    const int H = ab.n_steps;
    V3 pn, wn;        // position and body rate after the step in hand
    Q4 q0;            // unit attitude at step 0
    const size_t row = 4 * ns;
    if (FULL_TAPE) {
      const float4* const tape = ab.tape + slot;
      {
        const float4* e = tape + (size_t)H * row;
        const float4 e0 = e[0], e1 = e[ns], e3 = e[3 * ns];
        pn = {e0.x, e0.y, e0.z};
        wn = {e1.z, e1.w, e3.x};
      }
      auto request = [&](int t) {  // a group per step, empty before the first
        if (t >= 0) {
          const float4* e = tape + (size_t)t * row;
#pragma unroll
          for (int r = 0; r < 4; ++r) copy16_async(&ring[t % kSweepStages][r][lane], e + r * ns);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
#pragma unroll
      for (int k = 1; k < kSweepStages; ++k) request(H - k);
      for (int t = H - 1; t >= 0; --t) {
        request(t - (kSweepStages - 1));
        asm volatile("cp.async.wait_group %0;" ::"n"(kSweepStages - 1) : "memory");
        const float4(*e)[kAdjointBlock] = ring[t % kSweepStages];
        const TapeStep x = unpack(e[0][lane], e[1][lane], e[2][lane], e[3][lane]);
        backward_step<NROT, MODE>(x, pn, wn, cm, b, P, goal, cp2, cw2, z, gb);
        pn = x.p;
        wn = x.w;
        q0 = x.q;
      }
    } else {
      const int K = ab.K;
      for (int seg = (H + K - 1) / K - 1; seg >= 0; --seg) {
        const int t0 = seg * K, len = H - t0 < K ? H - t0 : K;
        float4* const tape = ab.tape + slot;
        Vehicle<NROT> v;
        const float* ck = ab.ckpt + (size_t)seg * 21 * n;
        load_vehicle(ck, ck + 13 * n, (uint32_t)n, env, v);
        for (int t = 0; t < len; ++t) {
          const VState start = v.s;
          float wf;
          uint32_t pass = 0;
          forward_step<NROT, MODE>(v, cm, b, P, wf, pass);
          store_entry(tape + (size_t)t * row, ns, start, wf, pass);
        }
        if (t0 + len == H) {  // the later segments' first entries carry pn and wn across the others
          pn = v.s.p;
          wn = v.s.w;
        }
        for (int t = len - 1; t >= 0; --t) {
          const float4* e = tape + (size_t)t * row;
          const TapeStep x = unpack(e[0], e[ns], e[2 * ns], e[3 * ns]);
          backward_step<NROT, MODE>(x, pn, wn, cm, b, P, goal, cp2, cw2, z, gb);
          pn = x.p;
          wn = x.w;
          q0 = x.q;
        }
      }
    }
    // the rollout started from q_0 / |q_0|: the adjoint of q_0 is 2 q (0, g) / |q_0|
    const float s = 2.f * ab.inv_q0[slot];
    const Q4 qb = quat_rate2(q0, z.g);
    if (ab.grad_x0) {
      float* gx = ab.grad_x0 + env;
      const float v13[13] = {z.p.x, z.p.y, z.p.z, z.v.x, z.v.y, z.v.z, s * qb.w, s * qb.x, s * qb.y, s * qb.z,
                             z.w.x, z.w.y, z.w.z};
#pragma unroll
      for (int k = 0; k < 13; ++k) gx[k * n] = v13[k];
    }
    if (ab.grad_gains_env) {
      float* gg = ab.grad_gains_env + env;
      const float v12[12] = {gb.kx.x, gb.kx.y, gb.kx.z, gb.kv.x, gb.kv.y, gb.kv.z,
                             gb.kR.x, gb.kR.y, gb.kR.z, gb.kW.x, gb.kW.y, gb.kW.z};
#pragma unroll
      for (int k = 0; k < 12; ++k) gg[k * n] = v12[k];
    }
    if (ab.grad_targets) {
#pragma unroll
      for (int k = 0; k < 4; ++k) ab.grad_targets[k * n + env] = gb.tb[k];
    }
    gains[0] = gb.kx;
    gains[1] = gb.kv;
    gains[2] = gb.kR;
    gains[3] = gb.kW;
  }
};

// One warp per block and at most 128 registers: four warps fit per SM
// sub-partition, 16 per SM, so a 65,536-vehicle fleet (2,048 warps) is
// resident in one wave on 152 SMs; three words spill. Bound by instruction issue
// (72 % of cycles, and the sub-partitions that hold four warps, not three,
// finish last); the tape leaves DRAM at half its rate. 65,536 quads x 256
// steps: 267 us for 202 M warp instructions, against 501 us for 365 M (and
// 194 us for a launch that recomputed the tape) when the sweep rebuilt the
// whole step and carried the adjoints of q and R.
// The warp's sum of each gain's adjoint (a fixed tree over its lanes) goes to
// partial[gain][warp].
template <bool FULL_TAPE>
__global__ void __maxnreg__(128) k_adjoint(AdjointBuffers ab, StepParams P) {
  __shared__ float4 ring[FULL_TAPE ? kSweepStages : 1][4][kAdjointBlock];
  const uint32_t slot = blockIdx.x * kAdjointBlock + threadIdx.x;
  V3 gains[4] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  const uint32_t env = ab.order[slot];  // n_slots is a multiple of the block
  if (env < ab.n)
    by_airframe_and_mode(rotors_of(ab, env), mode_of(ab, env), Sweep<FULL_TAPE>{ab, P, slot, env, ring, gains});
  __syncwarp();
  const float v12[12] = {gains[0].x, gains[0].y, gains[0].z, gains[1].x, gains[1].y, gains[1].z,
                         gains[2].x, gains[2].y, gains[2].z, gains[3].x, gains[3].y, gains[3].z};
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    float v = v12[k];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    if (threadIdx.x == 0) ab.partial[(size_t)k * gridDim.x + blockIdx.x] = v;
  }
}

// Fleet sum of the warps' partial sums: one block per gain, each thread over a
// fixed stride, then a fixed tree, so repeated calls give identical bits.
constexpr int kRedThreads = 1024;
__global__ void __launch_bounds__(kRedThreads) k_reduce_gains(const float* partial, uint32_t parts, float* out) {
  __shared__ float sh[kRedThreads / 32];
  const float* p = partial + (size_t)blockIdx.x * parts;
  float acc = 0.f;
  for (uint32_t j = threadIdx.x; j < parts; j += kRedThreads) acc += p[j];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, d);
  if ((threadIdx.x & 31u) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = sh[threadIdx.x];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    if (threadIdx.x == 0) out[blockIdx.x] = v;
  }
}

}  // namespace

cudaError_t launch_record(const AdjointBuffers& ab, const StepParams& P, cudaStream_t st) {
  const unsigned blocks = ab.n_slots / kRecordBlock;
  if (ab.full_tape) k_record<true><<<blocks, kRecordBlock, 0, st>>>(ab, P);
  else k_record<false><<<blocks, kRecordBlock, 0, st>>>(ab, P);
  return cudaGetLastError();
}

cudaError_t launch_adjoint(const AdjointBuffers& ab, const StepParams& P, cudaStream_t st) {
  const unsigned blocks = ab.n_slots / kAdjointBlock;
  if (ab.full_tape) k_adjoint<true><<<blocks, kAdjointBlock, 0, st>>>(ab, P);
  else k_adjoint<false><<<blocks, kAdjointBlock, 0, st>>>(ab, P);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !ab.grad_gains) return e;
  k_reduce_gains<<<12, kRedThreads, 0, st>>>(ab.partial, blocks, ab.grad_gains);
  return cudaGetLastError();
}

}  // namespace agk
