// The device-side bookkeeping of a step, shared by the step kernels and the
// persistent 1D run.
#pragma once

#include <cuda_runtime.h>

#include "enoao.h"
#include "enoao_internal.h"

namespace enoao {

struct StepConsts {
  int system, ndim;
  int field;  // per-field splitting constants (Euler)
  double adv_speed;
  double dx[3];
};

__device__ inline void finalize_pending(StepState* st) {
  if (st->err & kErrBarrier) st->pending = 0;
  if (st->pending) {
    st->t = st->last ? st->t_end : st->t + st->dt;
    st->steps += 1;
    if (st->last) st->done = 1;
    st->pending = 0;
  }
}

// Per-field constants of the step from the running maxima of slot cur (the
// one-alpha value, for dt, is the largest of them); clear: the other slot too.
// alpha of axis d for the CFL rule (Euler): |u_d| + c of slot cur, which per
// field is the larger of max |u_d - c| and max |u_d + c| (the last stage then
// accumulates only the per-field maxima).
__device__ inline double step_alpha(const StepState* st, const StepConsts& k, int cur, int d) {
  if (k.field)
    return fmax(__longlong_as_double((long long)st->alpha_acc_f[cur][d][0]),
                __longlong_as_double((long long)st->alpha_acc_f[cur][d][2]));
  return __longlong_as_double((long long)st->alpha_acc[cur][d]);
}

__device__ inline void load_field_alpha(StepState* st, const StepConsts& k, int cur, bool clear) {
  if (!k.field) return;
  for (int d = 0; d < 3; ++d)
    for (int f = 0; f < 3; ++f) {
      st->alpha_f[d][f] = d < k.ndim ? __longlong_as_double((long long)st->alpha_acc_f[cur][d][f]) : 0.0;
      if (clear) st->alpha_acc_f[cur ^ 1][d][f] = 0ull;
    }
}

// Start of a step: finalise the previous one, fix alpha from U^n and dt from
// the CFL rule (or the fixed step), shortened to land on t_end.
__device__ inline void begin_step(StepState* st, const StepConsts& k) {
  finalize_pending(st);
  if (st->done || (st->max_steps > 0 && st->steps >= st->max_steps) || st->err) {
    st->skip = 1;
    return;
  }
  st->skip = 0;
  const int cur = (int)(st->steps & 1);
  double s = 0.0;
  for (int d = 0; d < k.ndim; ++d) {
    const double a = k.system == ENOAO_EULER
                         ? step_alpha(st, k, cur, d)
                         : fabs(k.adv_speed);
    st->alpha[d] = a;
    s += a / k.dx[d];
  }
  st->par = cur ^ 1;
  for (int d = 0; d < 3; ++d) st->alpha_acc[cur ^ 1][d] = st->alpha_stage[d] = 0ull;
  load_field_alpha(st, k, cur, true);
  double dt = st->dt_fixed > 0.0 ? st->dt_fixed : st->cfl / s;
  st->last = 0;
  if (st->t + dt >= st->t_end) {
    dt = st->t_end - st->t;
    st->last = 1;
  }
  st->dt = dt;
  st->pending = 1;
}

}  // namespace enoao
