// Restarted mixed-precision GMRES on T_0 (per-step solve of the MOT recurrence).
#pragma once
#include "internal.h"

namespace tdc {
struct StepPlan;
struct GmresPlan;
cudaError_t build_gmres(tdcfie_t h, StepPlan* p);
void destroy_gmres(GmresPlan* g);
cudaError_t reset_gmres_stats(GmresPlan* g, cudaStream_t s);
void gmres_set_tol(GmresPlan* g, double tol);
// out5: Arnoldi iterations, steps, max per step, (unused), solves not converged
cudaError_t gmres_stats(GmresPlan* g, long long* out5);
// b: right-hand side (path type, R x ld); learned: learned guess buffer (or nullptr); T0p: T_0 in the
// path precision; solves step n = ctl->n + off into ring slot n % ring (one kernel).
template <typename T>
cudaError_t launch_gmres(tdcfie_t h, StepPlan* p, const T* b, const T* learned, const T* T0p, T* ringbuf, int off,
                         cudaStream_t s);

// Learned initial guess (mlp.cu): FP16 weights on the device, filled into p->guessbuf each step.
struct MlpState;
cudaError_t build_mlp(StepPlan* p, cudaStream_t s);
void destroy_mlp(MlpState* m);
cudaError_t mlp_load(StepPlan* p, const float* host_params, cudaStream_t s);
template <typename T>
int launch_mlp_guess(StepPlan* p, int off, cudaStream_t s);     // of step ctl->n + off; kernels enqueued
}  // namespace tdc
