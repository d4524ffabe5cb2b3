// Fixed-set CG loops of medium grids in one cooperative launch (coop.cuh).
#include "coop.cuh"

namespace bem {
size_t coop_shared_bytes() { return sizeof(CoopShared); }
cudaError_t launch_coop_cg(const CoopArgs& r, int lm, int lp, cudaStream_t s) {
  return launch_coop_kind<false>(r, lm, lp, s);
}
cudaError_t coop_setup_cg() { return coop_setup_kind<false>(); }
}  // namespace bem
