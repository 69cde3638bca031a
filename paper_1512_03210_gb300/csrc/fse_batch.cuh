// fse_batch.cuh -- the batched passes: run descriptors and launchers (see fse_batch.cu).
#pragma once

#include "fse_launch.cuh"

namespace fse {

struct BatchRun {
  void* psi;
  void* spec;
  const void* kin_half;
  const void* kin_full;
  double dt, omega, gx2, gy2;
  float beta_dt, lam, a0;  // beta dt, lambda, and dt over the kernel pass's lengths
};

// One pass of every run of a group (grid.y = run): a column pass along y of n
// points (VAR: COL_KIN2 on psi, COL_KHAT2 on the spectrum), an x pass of a kind.
// Phase passes read the trap's coefficients (x^2, y^2, x y) of their step from a
// table [step][run] that launch_batch_trap fills for up to kTrapSteps steps.
constexpr int kTrapSteps = 64;
cudaError_t launch_batch_trap(const BatchRun* runs, int nr, const double* t0, int step0, int nsteps, float4* trap,
                              cudaStream_t st);
template <int VAR>
cudaError_t launch_colb(int n, const ColArgs& a, const MulArgs& m, const void* tw, const BatchRun* runs, int nr,
                        int kin_full, cudaStream_t st);
cudaError_t launch_xb(int kind, int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const float4* trap, cudaStream_t st);

}  // namespace fse
