// Pass B of the FP64 path (64-bit block fixed point), and its tables.
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

// Twiddles as two 30-bit limbs per component (fx_kernels.cuh) from their FP64
// values: w 2^60 = h 2^30 + l, l in [-2^29, 2^29).
__global__ void k_fx_tables(const double2* __restrict__ w, int4* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double2 v = w[i];
    int4 q;
    const ll x = __double2ll_rn(v.x * 1152921504606846976.0), y = __double2ll_rn(v.y * 1152921504606846976.0);
    fsplit(x, q.x, q.y);
    fsplit(y, q.z, q.w);
    out[i] = q;
  }
}
void launch_fx_tables(const double2* w, int4* out, int n, cudaStream_t s) {
  k_fx_tables<<<std::min((n + 255) / 256, 128), 256, 0, s>>>(w, out, n);
}

}  // namespace bem
