// Polonsky-Keer loops of small grids in one cluster (resident.cuh).
#include "resident.cuh"

namespace bem {
cudaError_t launch_resident_pk(const ResArgs& r, int lm, int lp, int n, cudaStream_t s) {
  return launch_resident_kind<true>(r, lm, lp, n, s);
}
cudaError_t resident_setup_pk(bool* runs) {
  const cudaError_t e = resident_setup_kind<true>();
  *runs = e == cudaSuccess && resident_runs_kind<true>();
  return e;
}
}  // namespace bem
