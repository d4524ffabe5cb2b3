// Pass B of the FP64 path (64-bit block fixed point).
#include "fx_kernels.cuh"

namespace bem {

void launch_fx_b(const PassArgs<double>& a, const PassArgs<double>* arr, int n, cudaStream_t s) {
  const dim3 grid(a.pl.gridB, n), block(a.pl.threadsB);
  switch (a.pl.gB.logL) {
#define BEM_CASE(LG)                                                    \
  case LG:                                                              \
    if (arr) k_fx_b_mi<LG><<<grid, block, a.pl.smemB, s>>>(arr);        \
    else k_fx_b<LG><<<grid, block, a.pl.smemB, s>>>(a);                 \
    break;
    BEM_LOGL_CASES_B(BEM_CASE)
#undef BEM_CASE
  }
}

cudaError_t set_smem_attrs_fx_b(int bytes) {
  cudaError_t e = cudaSuccess, r;
#define BEM_ATTR(fn) \
  if ((r = set_smem_max(fn, bytes)) != cudaSuccess && e == cudaSuccess) e = r;
#define BEM_CASE(LG) BEM_ATTR((k_fx_b<LG>)) BEM_ATTR((k_fx_b_mi<LG>))
  BEM_LOGL_CASES_B(BEM_CASE)
#undef BEM_CASE
#undef BEM_ATTR
  return e;
}

}  // namespace bem
