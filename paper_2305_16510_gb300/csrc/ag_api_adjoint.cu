// ag_api_adjoint.cu — extern "C" entry points of the differentiable rollout
// (ag_set_gains, ag_rollout_loss, ag_backward).
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>

#include <cuda_runtime.h>

#include "ctx_internal.h"

using namespace agh;

// ---------------------------------------------------------------------------
// Differentiable rollout: gains, recorded forward, adjoint.
namespace {

// Buffers of a record of n_steps steps with checkpoint interval K: the tape of
// the whole horizon when it fits (within hbm_budget_bytes when one is set), so
// that the record writes what the sweep reads; else a tape of one segment and
// the checkpoints the sweep recomputes it from.
ag_status ensure_adjoint(ag_ctx* ctx, int n_steps, int K) {
  agk::AdjointBuffers& a = ctx->adj;
  const size_t n = ctx->cfg.n_envs, slots = ctx->fb.n_slots;
  const size_t n_ckpt = (size_t)(n_steps + K - 1) / K;
  cudaError_t e = cudaSuccess;
  if (!a.loss) {
    const size_t bytes_before = ctx->bytes;
    float* pg = nullptr; float* lw = nullptr;
    if (e == cudaSuccess) e = alloc(ctx, &pg, 3 * n);
    if (e == cudaSuccess) e = alloc(ctx, &a.saturated, n);
    if (e == cudaSuccess) e = alloc(ctx, &lw, n);
    if (e == cudaSuccess) e = alloc(ctx, &a.inv_q0, slots);
    if (e == cudaSuccess) e = alloc(ctx, &a.grad_x0, 13 * n);
    if (e == cudaSuccess) e = alloc(ctx, &a.grad_gains_env, 12 * n);
    if (e == cudaSuccess) e = alloc(ctx, &a.grad_targets, 4 * n);
    if (e == cudaSuccess) e = alloc(ctx, &a.partial, 12 * (slots / 32));
    if (e == cudaSuccess) e = alloc(ctx, &a.grad_gains, 12);
    a.p_goal = pg;
    a.loss_weights = lw;
    if (e == cudaSuccess) e = alloc(ctx, &a.loss, slots);  // as long as the order: see keep_recorded_order
    if (e != cudaSuccess) {  // nothing half-allocated stays: the next call starts over
      cudaGetLastError();
      void* got[] = {(void*)a.p_goal, a.saturated, (void*)a.loss_weights, a.inv_q0, a.grad_x0, a.grad_gains_env,
                     a.grad_targets, a.partial, a.grad_gains};
      for (void* p : got)
        if (p) cudaFree(p);
      a = agk::AdjointBuffers{};
      ctx->bytes = bytes_before;
      ctx->err = "adjoint buffers do not fit";
      return AG_ERR_OOM;
    }
  }
  const size_t entry_bytes = agk::kTapeWords * slots * sizeof(float4);
  const size_t held = (size_t)ctx->adj_tape_cap * entry_bytes;
  auto free_tape = [&]() {
    if (a.tape) {
      cudaStreamSynchronize(ctx->stream);
      cudaFree(a.tape);
      a.tape = nullptr;
      ctx->bytes -= held;
    }
    ctx->adj_tape_cap = 0;
  };
  const size_t full = (size_t)n_steps + 1;  // one entry per step and the end state
  if (ctx->adj_tape_cap < full) {
    if (agk::tape_within_budget(ctx->cfg.hbm_budget_bytes, ctx->bytes - held, full, slots)) {
      free_tape();
      if (alloc(ctx, &a.tape, full * agk::kTapeWords * slots) == cudaSuccess) {
        ctx->adj_tape_cap = full;
      } else {
        cudaGetLastError();  // an out-of-memory cudaMalloc leaves no sticky error
        a.tape = nullptr;
      }
    }
  }
  a.full_tape = ctx->adj_tape_cap >= full ? 1 : 0;
  if (a.full_tape) return AG_OK;
  const size_t entries = (size_t)(K < n_steps ? K : n_steps);
  if (entries > ctx->adj_tape_cap) {
    free_tape();
    e = alloc(ctx, &a.tape, entries * agk::kTapeWords * slots);
    if (e != cudaSuccess) { cudaGetLastError(); a.tape = nullptr; ctx->err = "tape does not fit"; return AG_ERR_OOM; }
    ctx->adj_tape_cap = entries;
  }
  if (n_ckpt > ctx->adj_ckpt_cap) {
    if (a.ckpt) {
      cudaStreamSynchronize(ctx->stream);
      cudaFree(a.ckpt);
      a.ckpt = nullptr;
      ctx->bytes -= ctx->adj_ckpt_cap * 21 * n * sizeof(float);
      ctx->adj_ckpt_cap = 0;
    }
    e = alloc(ctx, &a.ckpt, n_ckpt * 21 * n);
    if (e != cudaSuccess) { cudaGetLastError(); a.ckpt = nullptr; ctx->err = "checkpoints do not fit"; return AG_ERR_OOM; }
    ctx->adj_ckpt_cap = n_ckpt;
  }
  return AG_OK;
}

bool overlap(const float* a, size_t na, const float* b, size_t nb) { return a < b + nb && b < a + na; }

}  // namespace

namespace agh {

ag_status keep_recorded_order(ag_ctx* ctx) {
  agk::AdjointBuffers& a = ctx->adj;
  if (!ctx->adj_recorded || a.order != ctx->fb.order) return AG_OK;
  // the copies lie in the staging of the loss and the flags, which nothing reads between a record's end and the next
  ag_status s = check_cuda(ctx, cudaMemcpyAsync(a.loss, a.order, a.n_slots * sizeof(uint32_t), cudaMemcpyDeviceToDevice,
                                                ctx->stream), "keep order");
  if (s == AG_OK)
    s = check_cuda(ctx, cudaMemcpyAsync(a.saturated, a.modes, a.n, cudaMemcpyDeviceToDevice, ctx->stream), "keep modes");
  if (s != AG_OK) return s;
  a.order = reinterpret_cast<const uint32_t*>(a.loss);
  a.modes = a.saturated;
  return AG_OK;
}

}  // namespace agh

extern "C" ag_status ag_set_gains(ag_ctx* ctx, const float* gains12) {
  ag_status s = enter(ctx);
  if (s != AG_OK) return s;
  if (!gains12) return fail_invalid(ctx, "gains is NULL");
  float g[12];
  if (on_host(gains12)) {
    std::memcpy(g, gains12, sizeof(g));  // no CUDA call: a synchronous cudaMemcpy waits for the device's queued work
  } else if ((s = check_cuda(ctx, cudaMemcpy(g, gains12, sizeof(g), cudaMemcpyDefault), "copy gains")) != AG_OK) {
    return s;
  }
  for (int i = 0; i < 12; ++i)
    if (!std::isfinite(g[i])) return fail_invalid(ctx, "gains must be finite");
  for (int i = 0; i < 3; ++i) {
    ctx->cfg.kx[i] = g[i]; ctx->cfg.kv[i] = g[3 + i]; ctx->cfg.kR[i] = g[6 + i]; ctx->cfg.kW[i] = g[9 + i];
  }
  return AG_OK;
}

extern "C" ag_status ag_rollout_loss(ag_ctx* ctx, uint32_t n_steps, float w_pos, float w_omega, const float* p_goal,
                                     float* loss, uint8_t* saturated) {
  agk::NvtxRange range("ag_rollout_loss");
  ag_status s = enter(ctx);
  if (s != AG_OK) return s;
  const ag_config& c = ctx->cfg;
  if (c.integrator != AG_INTEG_SIE || c.substeps_per_step != 1 || c.n_obstacles != 0) {
    ctx->err = "the differentiable rollout needs semi-implicit Euler, 1 substep per step and no obstacles";
    return AG_ERR_UNSUPPORTED;
  }
  if (n_steps == 0 || n_steps > (1u << 30) || !p_goal || !loss)
    return fail_invalid(ctx, "n_steps must be in 1..2^30; p_goal and loss are required");
  const size_t n = c.n_envs;
  const int K = c.record_every ? (int)c.record_every : 32;
  ctx->adj_recorded = false;  // the buffers of the last record may be replaced
  if ((s = ensure_adjoint(ctx, (int)n_steps, K)) != AG_OK) return s;
  agk::AdjointBuffers& a = ctx->adj;
  // goals and loss in the context's own device memory are read and written in place
  const bool loss_here = on_own_device(ctx, loss);
  a.goal_in = p_goal;
  if (!on_own_device(ctx, p_goal) || (loss_here && overlap(loss, n, p_goal, 3 * n))) {
    if ((s = check_cuda(ctx, cudaMemcpyAsync(a.p_goal, p_goal, 3 * n * sizeof(float), cudaMemcpyDefault, ctx->stream),
                        "copy goals")) != AG_OK) return s;
    a.goal_in = a.p_goal;
  }
  a.state = ctx->fb.state; a.motors = ctx->fb.motors; a.body = ctx->fb.body; a.targets = ctx->fb.targets;
  a.modes = ctx->fb.modes;
  a.order = ctx->fb.order;
  a.n_slots = ctx->fb.n_slots;
  a.n = c.n_envs; a.n_quad = c.n_quad; a.n_hexa = c.n_hexa; a.n_octo = c.n_octo;
  a.n_steps = (int)n_steps; a.K = K; a.w_pos = w_pos; a.w_omega = w_omega;
  ctx->adj_P = step_params(ctx);
  agk::AdjointBuffers rec = a;
  if (loss_here) rec.loss = loss;
  a.goal_in = nullptr;  // the caller's array is not read after this launch
  if ((s = check_cuda(ctx, agk::launch_record(rec, ctx->adj_P, ctx->stream), "record launch")) != AG_OK) return s;
  ctx->adj_recorded = true;
  if (!loss_here && (s = check_cuda(ctx, cudaMemcpyAsync(loss, a.loss, n * sizeof(float), cudaMemcpyDefault, ctx->stream),
                                 "copy loss out")) != AG_OK) return s;
  if (saturated)
    s = check_cuda(ctx, cudaMemcpyAsync(saturated, a.saturated, n, cudaMemcpyDefault, ctx->stream), "copy flags out");
  return s;
}

extern "C" ag_status ag_backward(ag_ctx* ctx, const float* loss_weights, float* grad_x0, float* grad_gains,
                                 float* grad_gains_per_env, float* grad_targets) {
  agk::NvtxRange range("ag_backward");
  ag_status s = enter(ctx);
  if (s != AG_OK) return s;
  if (!ctx->adj_recorded) {
    ctx->err = "ag_backward needs a rollout recorded by ag_rollout_loss";
    return AG_ERR_STATE;
  }
  if (!grad_x0 && !grad_gains && !grad_gains_per_env && !grad_targets) return AG_OK;
  agk::AdjointBuffers a = ctx->adj;
  const size_t n = ctx->cfg.n_envs;
  // a wanted output in the context's own device memory is written in place, any other through the staging
  // buffer; unwanted ones are not formed
  struct Out { float* user; float** field; float* stage; size_t count; const char* what; };
  const Out outs[4] = {{grad_x0, &a.grad_x0, a.grad_x0, 13 * n, "copy grad x0"},
                       {grad_gains, &a.grad_gains, a.grad_gains, 12, "copy grad gains"},
                       {grad_gains_per_env, &a.grad_gains_env, a.grad_gains_env, 12 * n, "copy per-env grad gains"},
                       {grad_targets, &a.grad_targets, a.grad_targets, 4 * n, "copy grad targets"}};
  bool staged[4];
  for (int k = 0; k < 4; ++k) {
    staged[k] = outs[k].user && !on_own_device(ctx, outs[k].user);
    *outs[k].field = staged[k] ? outs[k].stage : outs[k].user;
  }
  // the weights are read in place where a copy is not needed
  bool weights_here = loss_weights && on_own_device(ctx, loss_weights);
  for (int k = 0; k < 4; ++k)
    if (weights_here && outs[k].user && overlap(outs[k].user, outs[k].count, loss_weights, n)) weights_here = false;
  if (loss_weights && !weights_here &&
      (s = check_cuda(ctx, cudaMemcpyAsync((void*)a.loss_weights, loss_weights, n * sizeof(float), cudaMemcpyDefault,
                                           ctx->stream), "copy weights")) != AG_OK)
    return s;
  if (!loss_weights || weights_here) a.loss_weights = loss_weights;
  if ((s = check_cuda(ctx, agk::launch_adjoint(a, ctx->adj_P, ctx->stream), "adjoint launch")) != AG_OK) return s;
  for (int k = 0; k < 4; ++k)
    if (staged[k] && (s = check_cuda(ctx, cudaMemcpyAsync(outs[k].user, outs[k].stage, outs[k].count * sizeof(float),
                                                          cudaMemcpyDefault, ctx->stream), outs[k].what)) != AG_OK)
      return s;
  return s;
}
