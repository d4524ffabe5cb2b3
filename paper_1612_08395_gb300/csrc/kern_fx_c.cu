// Pass C of the FP64 path (64-bit block fixed point) for every supported length.
#include "fx_kernels.cuh"

namespace bem {
template void launch_pass_c<double>(const PassArgs<double>&, int, cudaStream_t);
template void launch_pass_c_mi<double>(const PassArgs<double>&, int, const PassArgs<double>*, int, cudaStream_t);

void launch_fx_c(const PassArgs<double>& a, int mode, const PassArgs<double>* arr, int n, cudaStream_t s) {
  switch (mode) {
    case C_PLAIN: launch_fx_c_mode<C_PLAIN>(a, arr, n, s); break;
    case C_PK_G: launch_fx_c_mode<C_PK_G>(a, arr, n, s); break;
    case C_PK_R: launch_fx_c_mode<C_PK_R>(a, arr, n, s); break;
    case C_CG_R: launch_fx_c_mode<C_CG_R>(a, arr, n, s); break;
    case C_CG_G: launch_fx_c_mode<C_CG_G>(a, arr, n, s); break;
    case C_GAP: launch_fx_c_mode<C_GAP>(a, arr, n, s); break;
  }
}

cudaError_t set_smem_attrs_fx_c(int bytes) {
  cudaError_t e = cudaSuccess, r;
#define BEM_ATTR(fn) \
  if ((r = set_smem_max(fn, bytes)) != cudaSuccess && e == cudaSuccess) e = r;
#define BEM_CASE(LG)                                                                          \
  BEM_ATTR((k_fx_c<C_PLAIN, LG>)) BEM_ATTR((k_fx_c<C_PK_G, LG>)) BEM_ATTR((k_fx_c<C_PK_R, LG>)) \
  BEM_ATTR((k_fx_c<C_CG_R, LG>)) BEM_ATTR((k_fx_c<C_CG_G, LG>)) BEM_ATTR((k_fx_c<C_GAP, LG>))   \
  BEM_ATTR((k_fx_c_mi<C_PK_G, LG>)) BEM_ATTR((k_fx_c_mi<C_PK_R, LG>)) BEM_ATTR((k_fx_c_mi<C_CG_R, LG>))
  BEM_LOGL_CASES_A(BEM_CASE)
#undef BEM_CASE
#undef BEM_ATTR
  return e;
}

}  // namespace bem
