// Fixed-set CG loops of small grids in one cluster (resident.cuh).
#include "resident.cuh"

namespace bem {
cudaError_t launch_resident_cg(const ResArgs& r, int lm, int lp, int n, cudaStream_t s) {
  return launch_resident_kind<false>(r, lm, lp, n, s);
}
cudaError_t resident_setup_cg(bool* runs) {
  const cudaError_t e = resident_setup_kind<false>();
  *runs = e == cudaSuccess && resident_runs_kind<false>();
  return e;
}
}  // namespace bem
