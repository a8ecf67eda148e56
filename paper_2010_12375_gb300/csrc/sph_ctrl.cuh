// Acoustic time-step control of one substep (Eq. dt-relax), shared by the per-launch
// kernel (k_dt_acoustic) and the persistent substep loop.
#pragma once
#include "sph_common.cuh"

namespace sph {

// One tank's next acoustic substep: dt = min(cfl_ac h / (c0 + |v|max), Dt_ad - tau), tau and
// t advanced; the tank is done once its Dt_ad is covered, and a done tank gets dt = 0 (its
// particles sit this substep out). A non-finite or vanishing step sets ERR_DT, a substep
// count beyond the tank's bound ERR_TIMEOUT, and either ends the tank's loop instead of
// letting a device-side loop spin. cap: a cap on the acoustic step (0 = none). Returns
// whether the tank needs substeps after this one.
__device__ __forceinline__ int dt_acoustic_one(const Inst& I, Ctrl& C, Global* g, double cap) {
  if (C.done) {
    C.dt = 0.0;
    return 0;
  }
  double vmax = sqrt((double)__uint_as_float(C.vmax2));
  C.vmax2 = 0u;                                     // refilled by the pressure relaxation
  double dt_ac = I.cfl_ac * I.h_d / (I.c0_d + vmax);
  if (cap > 0.0) dt_ac = fmin(dt_ac, cap);
  double rem = C.dt_ad - C.tau;
  double dt = fmin(dt_ac, rem);
  if (!(dt_ac > I.dt_min) || !(rem > 0.0) || !(dt > 0.0)) {
    atomicOr(&g->err, ERR_DT);
    C.dt = 0.0;
    C.done = 1;
    return 0;
  }
  if (C.sub_in_step >= I.max_sub) {
    atomicOr(&g->err, ERR_TIMEOUT);
    C.dt = 0.0;
    C.done = 1;
    return 0;
  }
  C.dt = dt;
  C.tau += dt;
  C.t += dt;
  C.substeps += 1;
  C.sub_in_step += 1;
  if (C.tau >= C.dt_ad * (1.0 - kLoopSlack)) {
    C.done = 1;
    return 0;
  }
  return 1;
}

// Eq. dt-advection of one tank: Dt_ad = CFL_ad min(h / max(|v|max, U_ref), h^2 / nu), the
// start of its advection step.
__device__ __forceinline__ void dt_advection_one(const Inst& I, Ctrl& C) {
  double vmax = sqrt((double)__uint_as_float(C.vmax2));
  double dt = I.h_d / fmax(vmax, I.u_ref);
  if (I.nu > 0.0) dt = fmin(dt, I.h_d * I.h_d / I.nu);
  C.dt_ad = I.cfl_ad * dt;
  C.tau = 0.0;
  C.done = 0;
  C.dt = 0.0;
  C.sub_in_step = 0;
  C.adv_steps += 1;
}

// Run by all threads of one block: the next substep of every tank. Returns, in every thread,
// whether some tank still needs substeps after this one. dt_cap (or NULL): per tank, a cap on
// the acoustic step (0 = none), written by a coupled solid run with single time stepping.
__device__ __forceinline__ int dt_acoustic_block(int n_inst, const Inst* __restrict__ inst, Ctrl* ctrl, Global* g,
                                                 const double* dt_cap = nullptr) {
  int any = 0;
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x)
    any |= dt_acoustic_one(inst[k], ctrl[k], g, dt_cap ? dt_cap[k] : 0.0);
  return __syncthreads_or(any);
}

}  // namespace sph
