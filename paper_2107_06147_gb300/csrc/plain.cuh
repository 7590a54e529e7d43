// plain.cuh -- the plain per-step FP64 form: every time step is a sequence of separate kernels over the whole
// batch, with the wave functions in global memory between kernels:
//   space half-step + first pass | middle pass | last pass + kinetic factor + first pass | middle pass |
//   last pass + space half-step + norm | waiting-time test / jump.
// It computes the same step as the fused kernel (Sec. 3.3, steps 1-5) with the same sine transform (fused.cuh: the
// passes' exchange is a global array instead of shared memory), and is the baseline the fused forms are measured
// against and the FP64 form beyond N = 8192.
#pragma once
#include "fused_plan.h"
#include "qtraj_device.cuh"

namespace qt {

// per-trajectory state of the plain form, kept in global memory between the kernels of a step
struct PlainState {
    double thr, ul, uc, r0; // current waiting-time threshold and jump draws; first threshold
    int l, c, nj, fj, flags, active, kdraw, executed, lj;
    uint32_t digest;   // jump digest (qtraj_obs.jump_digest)
};

__device__ __forceinline__ bool plain_running(const PlainState &s, const TrajDev &d, int n)
{
    return s.active && n < d.n_steps;
}

struct PlainBuffers {
    cpx<double> *psi;        // [n_traj][N] states: value e of thread g at e G + g, with the odd extension's sign
    cpx<double> *sa, *sb;    // [n_traj][plain_seq(N)] the exchange arrays of the two transforms
    double *n2;              // [n_traj][plain_parts(N)] partial norms
    PlainState *st;          // [n_traj]
};

// values of an exchange array and partial norms per trajectory
size_t plain_seq(int N);
int plain_parts(int N);

// Enqueues the whole evolution of a.n_traj trajectories (max_steps = longest medium) on `stream`.
cudaError_t plain_run(const Tables<double> &tb, const LaunchArgs &a, int N, int max_steps, PlainBuffers buf,
                      cudaStream_t stream, int *launches);

// the kernels of n_steps steps of one grid size (plain_step.cuh; instantiated in plain_a.cu, plain_b.cu)
struct PlainOps {
    int seq, parts;
    cudaError_t (*step)(const Tables<double> &, const LaunchArgs &, PlainBuffers, int n, cudaStream_t);   // 5 kernels
};
const PlainOps *plain_ops_a(int N);
const PlainOps *plain_ops_b(int N);

} // namespace qt
