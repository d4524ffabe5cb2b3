// Pass A of the FP64 path (64-bit block fixed point) for every supported length.
#include "fx_kernels.cuh"

namespace bem {

void launch_fx_a(const PassArgs<double>& a, int mode, const PassArgs<double>* arr, int n, cudaStream_t s) {
  switch (mode) {
    case A_PLAIN: launch_fx_a_mode<A_PLAIN>(a, arr, n, s); break;
    case A_PK_P: launch_fx_a_mode<A_PK_P>(a, arr, n, s); break;
    case A_PK_T: launch_fx_a_mode<A_PK_T>(a, arr, n, s); break;
    case A_CG_T: launch_fx_a_mode<A_CG_T>(a, arr, n, s); break;
  }
}

cudaError_t set_smem_attrs_fx_a(int bytes) {
  cudaError_t e = cudaSuccess, r;
#define BEM_ATTR(fn) \
  if ((r = set_smem_max(fn, bytes)) != cudaSuccess && e == cudaSuccess) e = r;
#define BEM_CASE(LG)                                                                          \
  BEM_ATTR((k_fx_a<A_PLAIN, LG>)) BEM_ATTR((k_fx_a<A_PK_P, LG>)) BEM_ATTR((k_fx_a<A_PK_T, LG>)) \
  BEM_ATTR((k_fx_a<A_CG_T, LG>)) BEM_ATTR((k_fx_a_mi<A_PK_P, LG>)) BEM_ATTR((k_fx_a_mi<A_PK_T, LG>)) \
  BEM_ATTR((k_fx_a_mi<A_CG_T, LG>))
  BEM_LOGL_CASES_A(BEM_CASE)
#undef BEM_CASE
#undef BEM_ATTR
  return e;
}

}  // namespace bem
