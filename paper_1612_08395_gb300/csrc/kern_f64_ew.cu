// FP64 instantiation of the elementwise kernels and the FP64 helpers of the
// refinement sweep, twiddle and index tables.
#include <algorithm>
#include "conv_kernels.cuh"

namespace bem {
BEM_INSTANTIATE_EW(double)

// p64 += dscale * dp on S (FP32 correction), optionally projected onto p >= 0.
__global__ void k_refine_apply(double* p64, const float* dp, double dscale, const uint8_t* S,
                               int project, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (!S[i]) continue;
    double v = p64[i] + dscale * (double)dp[i];
    if (project && v < 0.0) v = 0.0;
    p64[i] = v;
  }
}
void launch_refine_apply(double* p64, const float* dp, double dscale, const uint8_t* S, int project,
                         size_t n, cudaStream_t s) {
  k_refine_apply<<<ew_grid(n), 256, 0, s>>>(p64, dp, dscale, S, project, n);
}

// The correction's data: c = scale g, p = t = 0.
__global__ void k_refine_rhs(const double* g, double scale, float* c, float* p, float* t, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    c[i] = (float)(scale * g[i]);
    p[i] = 0.f;
    t[i] = 0.f;
  }
}
void launch_refine_rhs(const double* g, double scale, float* c, float* p, float* t, size_t n, cudaStream_t s) {
  k_refine_rhs<<<ew_grid(n), 256, 0, s>>>(g, scale, c, p, t, n);
}

// out[0] = max |a|, out[1] = max |b| over S (NaN skipped), as FP64; acc: two
// words and a counter, zero before and after.
__global__ void k_max_abs2(const double* __restrict__ a, const double* __restrict__ b, const uint8_t* __restrict__ S,
                           size_t n, unsigned long long* acc, unsigned int* counter, double* out) {
  __shared__ unsigned long long red[32];
  __shared__ int lastflag;
  unsigned long long ma = 0, mb = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (!S[i]) continue;
    ma = max(ma, abs_bits(a[i]));
    mb = max(mb, abs_bits(b[i]));
  }
  ma = block_max(ma, red);
  mb = block_max(mb, red);
  if (threadIdx.x == 0) {
    if (ma) atomicMax(acc, ma);
    if (mb) atomicMax(acc + 1, mb);
  }
  if (!last_block_arrival(counter, &lastflag)) return;
  if (threadIdx.x == 0) {
    out[0] = __longlong_as_double((long long)atomicExch(acc, 0ull));
    out[1] = __longlong_as_double((long long)atomicExch(acc + 1, 0ull));
    *counter = 0;
  }
}
void launch_max_abs2(const double* a, const double* b, const uint8_t* S, size_t n, unsigned long long* acc,
                     unsigned int* counter, double* out, cudaStream_t s) {
  k_max_abs2<<<std::min(ew_grid(n), 304), 256, 0, s>>>(a, b, S, n, acc, counter, out);
}

// The solve's scalars, all but the sticky error word: by kernel argument, so no
// copy engine, pinned staging or host wait is involved.
__global__ void k_set_scalars(Scalars v, Scalars* sc) {
  for (int i = threadIdx.x; i < (int)(offsetof(Scalars, kerr) / 4); i += blockDim.x)
    reinterpret_cast<int*>(sc)[i] = reinterpret_cast<const int*>(&v)[i];
}
void launch_set_scalars(const Scalars& v, Scalars* sc, cudaStream_t s) { k_set_scalars<<<1, 32, 0, s>>>(v, sc); }

__global__ void k_to_f32(const double* src, float* dst, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}
void launch_to_f32(const double* src, float* dst, size_t n, cudaStream_t s) {
  k_to_f32<<<ew_grid(n), 256, 0, s>>>(src, dst, n);
}

// ---------------------------------------------------------------------------
// All tables of a context in one launch, one entry per thread.  An entry costs
// one FP64 sincospi, a few hundred issue slots of the FP64 pipe for a warp:
// spread over the chip the tables of a 4096-point torus take a few microseconds
// (as a few CTAs looping over them, 62 us per length; the transform that makes its
// own tables on each call, 200 x 251: 152 -> 42 us with the FP64 passes' change).
//
// Stage twiddles of a length 2^logL transform, stages in DIF order, tables
// concatenated.  FP64 and fixed point: the table of stage (R, s) holds every
// power, exp(-2 pi i o q/(R s)) at (q-1) s + o for q = 1..R-1 (offsets
// FftC::pow_off; fewer than 2^logL entries in all).  FP32: exp(-2 pi i o/(R s))
// for o < s (radix-8 offsets tw_off8); the butterflies form the powers.
// w 2^62 = h 2^31 + l (fx_kernels.cuh): l in [-2^30, 2^30), but where h would be
// +-2^31 (|w| within 2^-32 of 1), which a 32-bit integer and its negative cannot
// both hold: there h = +-(2^31 - 1) and l takes the rest (+-1 less one unit for w = +-1).
__device__ __forceinline__ void fx_limb(double v, int& h, int& l) {
  const long long x = __double2ll_rn(v * 4611686018427387904.0);
  const long long lo = ((int)x << 1) >> 1, m = 0x7fffffff;
  const long long hi = min(max((x - lo) >> 31, -m), m);
  h = (int)hi;
  l = (int)min(max(x - (hi << 31), -m), m);
}
__device__ __forceinline__ int4 fx_limbs(double2 v) {
  int4 q;
  fx_limb(v.x, q.x, q.y);
  fx_limb(v.y, q.z, q.w);
  return q;
}
__device__ __forceinline__ double2 unit(double turns) {  // exp(2 pi i turns)
  double sn, cs;
  sincospi(2.0 * turns, &sn, &cs);
  return make_double2(cs, sn);
}
__device__ void stage_entry(int i, int logL, double2* t64, float2* t32, int4* fx) {
  const int r0 = logL % 3;
  int R = r0 ? (1 << r0) : 8, s = (1 << logL) / R, off = 0, off64 = 0;
  while (i - off64 >= (R - 1) * s) {  // the stage of entry i
    if (s == 1) return;
    off += s;
    off64 += (R - 1) * s;
    R = 8;
    s /= 8;
  }
  const int q = (i - off64) / s + 1, o = (i - off64) - (q - 1) * s;  // o q < R s
  const double2 w = unit(-(double)(o * q) / ((double)R * (double)s));
  if (t64) t64[i] = w;
  if (fx) fx[i] = fx_limbs(w);
  if (t32 && q == 1) t32[off + o] = make_float2((float)w.x, (float)w.y);
}
// FP32 stage tables of the radix-16 column pass of length 2^logL (9 <= logL <=
// 13; other lengths have none): a leading stage of radix 2^(logL mod 4) (16 if
// that is 1), then radix-16 stages; stage (R, s) holds exp(-2 pi i o/(R s)), o < s.
__device__ void stage16_entry(int i, int logL, float2* t32) {
  if (logL < 9 || logL > 13) return;
  const int rb = logL & 3;
  int R = rb ? 1 << rb : 16, s = (1 << logL) / R, off = 0;
  while (s > 1) {
    if (i < off + s) {
      const double2 w = unit(-(double)(i - off) / ((double)R * (double)s));
      t32[i] = make_float2((float)w.x, (float)w.y);
      return;
    }
    off += s;
    R = 16;
    s /= 16;
  }
}
// Index table of one transform length: sp[k] = swz(dig_pos(k)) (see Geo).
__device__ void geo_entry(int i, int* sp, const Geo& g, int esize) {
  const Swz z{g.sa, g.sb, g.sc, g.sd};
  const int x = dig_pos(i, g.logL, g.r0);
  sp[i] = esize == 4 ? swz<float>(x, z) : swz<double>(x, z);
}
__global__ void k_tables(TableArgs a) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int M = 1 << a.logM, P = 1 << a.logP;
  if (i < M) return stage_entry(i, a.logM, a.t64, a.t32, a.fx);
  i -= M;
  if (i < P)
    return stage_entry(i, a.logP, a.t64 ? a.t64 + M : nullptr, a.t32 ? a.t32 + M : nullptr, a.fx ? a.fx + M : nullptr);
  i -= P;
  if (i <= M) {  // exp(-i pi k / M): the real-FFT split
    const double2 w = unit(-0.5 * (double)i / (double)M);
    if (a.t64) a.t64[M + P + i] = w;
    if (a.t32) a.t32[M + P + i] = make_float2((float)w.x, (float)w.y);
    if (a.fx) a.fx[M + P + i] = fx_limbs(w);
    return;
  }
  i -= M + 1;
  if (a.t32) {
    if (i < P) return stage16_entry(i, a.logP, a.t32 + M + P + M + 1);
    i -= P;
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (!a.geo[t]) continue;
    const int n = 1 << a.g[t].logL;
    if (i < n) return geo_entry(i, a.geo[t], a.g[t], a.esize[t]);
    i -= n;
  }
}
void launch_tables(const TableArgs& a, cudaStream_t s) {
  const int M = 1 << a.logM, P = 1 << a.logP;
  int n = M + P + M + 1 + (a.t32 ? P : 0);
  for (int t = 0; t < 4; ++t)
    if (a.geo[t]) n += 1 << a.g[t].logL;
  k_tables<<<(n + 63) / 64, 64, 0, s>>>(a);
}

// Bounding box of the contact set: first/last row and column holding an
// element of S (atomicMin / atomicMax on sc->band0/band1/col0/col1, which start
// at ny / -1 / nx / -1).
__global__ void k_box(int nx, int ny, const uint8_t* S, Scalars* sc) {
  __shared__ int lo, hi, clo, chi;
  if (threadIdx.x == 0) { lo = ny; hi = -1; clo = nx; chi = -1; }
  __syncthreads();
  const bool vec = (nx & 15) == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
  int cmin = nx, cmax = -1;
  for (int row = blockIdx.x; row < ny; row += gridDim.x) {  // the same trip count in every thread
    const uint8_t* r = S + (size_t)row * nx;
    bool any = false;
    if (vec) {
      const uint4* r4 = reinterpret_cast<const uint4*>(r);
      for (int j = threadIdx.x; j < (nx >> 4); j += blockDim.x) {
        const uint4 v = r4[j];
        if ((v.x | v.y | v.z | v.w) != 0u) {
          any = true;
          for (int q = 0; q < 16; ++q)
            if (r[16 * j + q]) { cmin = min(cmin, 16 * j + q); cmax = max(cmax, 16 * j + q); }
        }
      }
    } else {
      for (int j = threadIdx.x; j < nx; j += blockDim.x)
        if (r[j]) { any = true; cmin = min(cmin, j); cmax = max(cmax, j); }
    }
    if (__syncthreads_or(any) && threadIdx.x == 0) {
      lo = min(lo, row);
      hi = max(hi, row);
    }
  }
  if (cmax >= 0) { atomicMin(&clo, cmin); atomicMax(&chi, cmax); }
  __syncthreads();
  if (threadIdx.x == 0 && hi >= 0) {
    atomicMin(&sc->band0, lo);
    atomicMax(&sc->band1, hi);
    atomicMin(&sc->col0, clo);
    atomicMax(&sc->col1, chi);
  }
}
// Bounding box of the geometric overlap set {h <= d} (into sc->band0/band1/
// col0/col1, which start at ny / -1 / nx / -1).
__global__ void k_box_overlap(int nx, int ny, const double* __restrict__ h, double d, Scalars* sc) {
  __shared__ int lo, hi, clo, chi;
  if (threadIdx.x == 0) { lo = ny; hi = -1; clo = nx; chi = -1; }
  __syncthreads();
  int cmin = nx, cmax = -1;
  for (int row = blockIdx.x; row < ny; row += gridDim.x) {  // the same trip count in every thread
    const double* r = h + (size_t)row * nx;
    bool any = false;
    for (int j = threadIdx.x; j < nx; j += blockDim.x)
      if (r[j] <= d) { any = true; cmin = min(cmin, j); cmax = max(cmax, j); }
    if (__syncthreads_or(any) && threadIdx.x == 0) {
      lo = min(lo, row);
      hi = max(hi, row);
    }
  }
  if (cmax >= 0) { atomicMin(&clo, cmin); atomicMax(&chi, cmax); }
  __syncthreads();
  if (threadIdx.x == 0 && hi >= 0) {
    atomicMin(&sc->band0, lo);
    atomicMax(&sc->band1, hi);
    atomicMin(&sc->col0, clo);
    atomicMax(&sc->col1, chi);
  }
}
void launch_box_overlap(const Plan& pl, const double* h, double d, Scalars* sc, cudaStream_t s) {
  const int grid = std::min(pl.ny, 2 * pl.nsm);
  k_box_overlap<<<grid, 256, 0, s>>>(pl.nx, pl.ny, h, d, sc);
}

// Copy the box [x0, x0+bx) x [y0, y0+by) of an nx x ny FP64 field, `fill` where
// the box leaves the grid (bx a power of two).
__global__ void k_box_copy64(const double* __restrict__ src, int nx, int ny, int x0, int y0,
                             double* __restrict__ dst, int lbx, int nb, double fill) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int X = x0 + (i & ((1 << lbx) - 1)), Y = y0 + (i >> lbx);
    dst[i] = (X < nx && Y < ny) ? src[(size_t)Y * nx + X] : fill;
  }
}
void launch_box_copy64(const double* src, int nx, int ny, int x0, int y0, double* dst, int bx, int by,
                       double fill, cudaStream_t s) {
  int lbx = 0;
  while ((1 << lbx) < bx) ++lbx;
  const int nb = bx * by;
  k_box_copy64<<<ew_grid((size_t)nb), 256, 0, s>>>(src, nx, ny, x0, y0, dst, lbx, nb, fill);
}

void launch_box(const Plan& pl, const uint8_t* S, Scalars* sc, cudaStream_t s) {
  const int grid = std::min(pl.ny, 2 * pl.nsm);
  k_box<<<grid, 256, 0, s>>>(pl.nx, pl.ny, S, sc);
}

__global__ void k_active_set(const double* p, const double* g, uint8_t* S, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    S[i] = (p[i] > 0.0 || g[i] < 0.0) ? 1 : 0;
}
void launch_active_set(const double* p, const double* g, uint8_t* S, size_t n, cudaStream_t s) {
  k_active_set<<<ew_grid(n), 256, 0, s>>>(p, g, S, n);
}
}  // namespace bem
