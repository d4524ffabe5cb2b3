// Fixed-set CG loops of medium grids in one cooperative launch (coop.cuh).
#include "coop.cuh"

namespace bem {
size_t coop_shared_bytes() { return sizeof(CoopShared); }
cudaError_t launch_coop_cg(const CoopArgs& r, int lm, int lp, cudaStream_t s) {
  return launch_coop_kind<false>(r, lm, lp, s);
}
// CTAs of the FP32 loops over `rows` rows (0: no kernel for these lengths, or too
// many rows for nsm SMs).
int coop_ctas(int lm, int lp, int rows, int nsm) {
  int nb = 0, R = 0;
  switch (lm * 16 + lp) {
#define BEM_CASE(LM, LP) case LM * 16 + LP: return coop_shape<LM, LP>(rows, nsm, &nb, &R) ? nb : 0;
    BEM_COOP_CASES(BEM_CASE)
#undef BEM_CASE
  }
  return 0;
}
cudaError_t coop_setup_cg() { return coop_setup_kind<false>(); }
}  // namespace bem
