// Influence coefficients K(di, dj) of Eq. 9 in FP64 on the device.
//
//   K(di, dj) = int_{(di-1/2)dx}^{(di+1/2)dx} int_{(dj-1/2)dy}^{(dj+1/2)dy} (a^2+b^2)^-(1+k)/2 db da
//
// Near the singularity (max(di, dj) <= NEAR) K is the corner difference of
//   F(x, y) = int_0^x int_0^y (a^2+b^2)^-(1+k)/2 db da
//           = [ x^(1-k) G(y/x) + y^(1-k) G(x/y) ] / (1-k),
//   G(U)    = int_0^{asinh U} cosh(s)^-k ds,
// obtained by integrating r^-(1+k) r dr exactly along rays from the corner
// (polar coordinates), then u = tan(theta) and u = sinh(s); the remaining
// integrand cosh^-k is smooth, so composite Gauss-Legendre converges fast.
// F is odd in each argument.  Away from the singularity the integrand is
// analytic on the element and tensor Gauss-Legendre rules are used directly,
// with fewer points the farther the element; the distance is counted in units
// of the element's longer side, so elongated elements near the singularity
// take the corner formula.  From SERIES sides on the element's mean is its
// Taylor series to sixth order in the sides (the eighth-order term is below
// 0.01 SERIES^-8 = 6e-17 of it), one power instead of sixteen: all but a corner
// of a large table.  Bound by FP64 instructions throughout.
//
// The corner formula takes a CTA per element and a thread per quadrature node,
// the tensor rules a warp per element: one thread evaluating an element's eight
// rays took 1.8 ms and its 256 nodes 0.6 ms, which every table, however small,
// had to wait for.  Square elements need half the table: K(di, dj) = K(dj, di).
// Together (GB300): 65^2 table 1.84 -> 0.04 ms, 1025^2 3.5 -> 0.1 ms.
#include <math.h>
#include <cuda_runtime.h>

#include "bem_impl.h"

namespace bem {

namespace {
constexpr int NG16 = 16;
constexpr int NEAR = 4;
constexpr int SERIES = 60;
__constant__ double c_x16[16], c_w16[16];
__constant__ double c_x10[10], c_w10[10];
__constant__ double c_x6[6], c_w6[6];

// Gauss-Legendre rule on [-1, 1]: roots of P_n by Newton's method, starting
// from the Tricomi approximation; P_n and P_n' from the Bonnet recurrence.
void legendre_rule(int n, double* x, double* w) {
  const double pi = 3.14159265358979323846;
  for (int i = 1; i <= n; ++i) {
    double th = pi * (4.0 * i - 1.0) / (4.0 * n + 2.0);
    double z = (1.0 - (n - 1.0) / (8.0 * n * n * n)) * cos(th);
    double dpn = 0.0;
    for (int it = 0; it < 60; ++it) {
      double pkm1 = 1.0, pk = z;
      for (int kk = 2; kk <= n; ++kk) {
        double pkp1 = ((2.0 * kk - 1.0) * z * pk - (kk - 1.0) * pkm1) / kk;
        pkm1 = pk;
        pk = pkp1;
      }
      dpn = n * (pkm1 - z * pk) / (1.0 - z * z);
      double step = pk / dpn;
      z -= step;
      if (fabs(step) <= 1e-16 * fabs(z) + 1e-300) break;
    }
    x[i - 1] = z;
    w[i - 1] = 2.0 / ((1.0 - z * z) * dpn * dpn);
  }
}
}  // namespace

int influence_init_nodes() {
  double x[16], w[16];
  legendre_rule(16, x, w);
  if (cudaMemcpyToSymbol(c_x16, x, sizeof(double) * 16) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(c_w16, w, sizeof(double) * 16) != cudaSuccess) return -1;
  legendre_rule(10, x, w);
  if (cudaMemcpyToSymbol(c_x10, x, sizeof(double) * 10) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(c_w10, w, sizeof(double) * 10) != cudaSuccess) return -1;
  legendre_rule(6, x, w);
  if (cudaMemcpyToSymbol(c_x6, x, sizeof(double) * 6) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(c_w6, w, sizeof(double) * 6) != cudaSuccess) return -1;
  return 0;
}

// distance class of the element: its index distance, but for elongated
// elements never more than its physical distance from the singularity in
// units of its longer side (a long element can reach close to the origin)
__device__ __forceinline__ double distance_class(int di, int dj, double dx, double dy) {
  const double ea = fmax(0.0, (di - 0.5) * dx), eb = fmax(0.0, (dj - 0.5) * dy);
  const double phys = sqrt(ea * ea + eb * eb) / fmax(dx, dy) + 0.5;
  return fmin((double)(di > dj ? di : dj), phys);
}

// The corner formula: K = F(a1, b1) - F(a0, b1) - F(a1, b0) + F(a0, b0), with
// F(x, y) = [ |x|^(1-k) G(|y/x|) + |y|^(1-k) G(|x/y|) ] / (1-k), odd in x and y,
// and G(U) = int_0^{asinh U} cosh(s)^-k ds by composite 16-point Gauss-Legendre
// with panels no longer than 0.5.  Thread t: corner t / 32, ray (t / 16) % 2,
// node t % 16 of every panel.
__global__ void __launch_bounds__(128) k_influence_near(double* Kq, int hx, int hy, double dx, double dy, double k) {
  const int di = blockIdx.x, dj = blockIdx.y;
  if (di >= hx || dj >= hy || distance_class(di, dj, dx, dy) > NEAR) return;
  __shared__ double part[8];
  const int c = threadIdx.x >> 5, ray = (threadIdx.x >> 4) & 1, i = threadIdx.x & 15;
  const double x = (di + (c & 1 ? 0.5 : -0.5)) * dx, y = (dj + (c & 2 ? 0.5 : -0.5)) * dy;
  const double p = fabs(ray ? y : x), q = fabs(ray ? x : y);
  double g = 0.0, hp = 0.0;
  if (p > 0.0 && q > 0.0) {
    const double S = asinh(q / p);
    const int np = max(1, (int)ceil(S / 0.5));
    hp = S / np;
    for (int m = 0; m < np; ++m) {
      const double s = (m + 0.5) * hp + 0.5 * hp * c_x16[i];
      g += exp(-k * log(cosh(s)));
    }
    g *= c_w16[i];
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
  if (i == 0) {
    double v = p > 0.0 && q > 0.0 ? pow(p, 1.0 - k) * (g * 0.5 * hp) / (1.0 - k) : 0.0;
    if ((x < 0.0) != (y < 0.0)) v = -v;
    part[threadIdx.x >> 4] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double F00 = part[0] + part[1], F10 = part[2] + part[3], F01 = part[4] + part[5], F11 = part[6] + part[7];
    Kq[(size_t)dj * hx + di] = F11 - F01 - F10 + F00;
  }
}

// Mean over the element of (x^2+y^2)^-a, a = (1+k)/2, times its area, by the
// Taylor series at its centre: with q = x^2+y^2, X = x^2/q, Y = y^2/q and
// c_n = a (a+1) ... (a+n-1), the derivative of order (2m, 2n) is q^-(a+m+n) times
// sum over j, i of (-1)^(m-j+n-i) A(m,j) A(n,i) c_(m+n+j+i) X^j Y^i,
// A(m,j) = 4^j (2m)! / ((m-j)! (2j)!); the mean takes it with
// (hx/2)^(2m) (hy/2)^(2n) / ((2m+1)! (2n+1)!).  Beyond 400 sides the sixth-order
// terms are below 3e-17 and left out.
__device__ __forceinline__ double series_mean(double x, double y, double hx, double hy, double k, bool sixth) {
  const double a = 0.5 * (1.0 + k);
  const double c1 = a, c2 = c1 * (a + 1.0), c3 = c2 * (a + 2.0), c4 = c3 * (a + 3.0), c5 = c4 * (a + 4.0),
               c6 = c5 * (a + 5.0);
  const double q = x * x + y * y, rq = 1.0 / q, X = x * x * rq, Y = y * y * rq;
  const double u = 0.25 * hx * hx * rq, v = 0.25 * hy * hy * rq;  // squared half sides over q
  const double xx = -2.0 * c1 + 4.0 * c2 * X, yy = -2.0 * c1 + 4.0 * c2 * Y;
  const double x4 = 12.0 * c2 + X * (-48.0 * c3 + 16.0 * c4 * X), y4 = 12.0 * c2 + Y * (-48.0 * c3 + 16.0 * c4 * Y);
  const double x2y2 = 4.0 * c2 - 8.0 * c3 + 16.0 * c4 * X * Y;
  const double s2 = (u * xx + v * yy) * (1.0 / 6.0);
  const double s4 = (u * u * x4 + v * v * y4) * (1.0 / 120.0) + u * v * x2y2 * (1.0 / 36.0);
  double s6 = 0.0;
  if (sixth) {
    const double x6 = -120.0 * c3 + X * (720.0 * c4 + X * (-480.0 * c5 + 64.0 * c6 * X));
    const double y6 = -120.0 * c3 + Y * (720.0 * c4 + Y * (-480.0 * c5 + 64.0 * c6 * Y));
    const double x4y2 = -24.0 * c3 + 48.0 * c4 * Y + X * (96.0 * c4 - 192.0 * c5 * Y + X * (-32.0 * c5 + 64.0 * c6 * Y));
    const double y4x2 = -24.0 * c3 + 48.0 * c4 * X + Y * (96.0 * c4 - 192.0 * c5 * X + Y * (-32.0 * c5 + 64.0 * c6 * X));
    s6 = (u * u * u * x6 + v * v * v * y6) * (1.0 / 5040.0) + u * v * (u * x4y2 + v * y4x2) * (1.0 / 720.0);
  }
  return hx * hy * exp(-a * log(q)) * (1.0 + (s2 + (s4 + s6)));
}

// One warp's sum of an element's NP x NP Gauss-Legendre nodes, in every lane.
template <int NP>
__device__ __forceinline__ double tensor_gl(const double* xs, const double* ws, double ca, double ha, double cb,
                                            double hb, double expo) {
  double s = 0.0;
  for (int q = threadIdx.x & 31; q < NP * NP; q += 32) {
    const int i = q / NP, j = q - i * NP;
    const double a = ca + ha * xs[i], b = cb + hb * xs[j];
    s += ws[i] * ws[j] * exp(expo * log(a * a + b * b));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s * ha * hb;
}
// Elements between the corner formula's and the series': a warp each, eight
// elements of one row per CTA.
__global__ void __launch_bounds__(256) k_influence_mid(double* Kq, int hx, int hy, double dx, double dy, double k) {
  const int di = blockIdx.x * 8 + (threadIdx.x >> 5), dj = blockIdx.y;
  if (di >= hx || dj >= hy) return;
  const double far = distance_class(di, dj, dx, dy);
  if (far <= NEAR || far > SERIES) return;
  const double expo = -0.5 * (1.0 + k);
  double v;
  if (far <= 12) v = tensor_gl<16>(c_x16, c_w16, di * dx, 0.5 * dx, dj * dy, 0.5 * dy, expo);
  else if (far <= 40) v = tensor_gl<10>(c_x10, c_w10, di * dx, 0.5 * dx, dj * dy, 0.5 * dy, expo);
  else v = tensor_gl<6>(c_x6, c_w6, di * dx, 0.5 * dx, dj * dy, 0.5 * dy, expo);
  if ((threadIdx.x & 31) == 0) Kq[(size_t)dj * hx + di] = v;
}

__global__ void k_influence(double* Kq, int hx, int hy, double dx, double dy, double k) {
  const int di = blockIdx.x * blockDim.x + threadIdx.x;
  const int dj = blockIdx.y;
  if (di >= hx || dj >= hy) return;
  const bool square = dx == dy;
  if (square && di < dj && dj < hx) return;  // written by the mirror element (its column dj is in the table)
  const double far = distance_class(di, dj, dx, dy);
  if (far <= SERIES) return;  // k_influence_near, k_influence_mid
  const double v = series_mean(di * dx, dj * dy, dx, dy, k, far <= 400.0);
  Kq[(size_t)dj * hx + di] = v;
  if (square && di > dj && di < hy) Kq[(size_t)di * hx + dj] = v;
}

// Elements whose distance class can be at most `far` along an axis of step d.
static int reach(double far, double side, double d, int n) {
  const double e = (far - 0.5) * side / d + 1.5;  // (i - 1/2) d <= (far - 1/2) side
  return e < n ? (int)e + 1 : n;
}

void launch_influence(double* Kq, int hx, int hy, double dx, double dy, double k, cudaStream_t s) {
  const double side = dx > dy ? dx : dy;
  const int nx = reach(NEAR, side, dx, hx), ny = reach(NEAR, side, dy, hy);
  k_influence_near<<<dim3(nx, ny), 128, 0, s>>>(Kq, hx, hy, dx, dy, k);
  const int mx = reach(SERIES, side, dx, hx), my = reach(SERIES, side, dy, hy);
  k_influence_mid<<<dim3((mx + 7) / 8, my), 256, 0, s>>>(Kq, hx, hy, dx, dy, k);
  if (mx == hx && my == hy && hx <= SERIES && hy <= SERIES) return;  // nothing farther
  const dim3 block(128), grid((hx + 127) / 128, hy);
  k_influence<<<grid, block, 0, s>>>(Kq, hx, hy, dx, dy, k);
}

}  // namespace bem
