// fse_batch.cuh -- the batched passes: run descriptors and launchers (see fse_batch.cu).
#pragma once

#include "fse_launch.cuh"

namespace fse {

struct BatchRun {
  void* psi;
  void* spec;
  const void* kin_half;
  const void* kin_full;
  double beta, lam, dt, omega, gx2, gy2;
};

// One pass of every run of a group (grid.y = run): a column pass along y of n
// points (VAR: COL_KIN2 on psi, COL_KHAT2 on the spectrum), an x pass of a kind.
template <int VAR>
cudaError_t launch_colb(int n, const ColArgs& a, const MulArgs& m, const void* tw,
                        const BatchRun* runs, int nr, int kin_full, cudaStream_t st);
cudaError_t launch_xb(int kind, int nx, const XArgs& a, const void* twn, const void* tw2n, const BatchRun* runs, int nr,
                      const double* t0, int step, cudaStream_t st);

}  // namespace fse
