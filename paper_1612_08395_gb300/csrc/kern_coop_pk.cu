// Polonsky-Keer loops of medium grids in one cooperative launch (coop.cuh).
#include "coop.cuh"

namespace bem {
cudaError_t launch_coop_pk(const CoopArgs& r, int lm, int lp, cudaStream_t s) {
  return launch_coop_kind<true>(r, lm, lp, s);
}
cudaError_t coop_setup_pk() { return coop_setup_kind<true>(); }
}  // namespace bem
