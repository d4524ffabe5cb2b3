// The FP64 path's transform passes in 64-bit block fixed point.
//
// GB300 issues FP64 arithmetic at about 2 operations per clock and SM (measured:
// 2.06 DFMA, 1.74 DADD) but 64-bit integer additions and 32 x 32 + 64 bit
// multiply-adds at about 60, so an FP64 FFT is bound by its instruction count at
// a thirtieth of the rate the same additions have in integers.  These kernels
// keep every value of a transform as a 64-bit integer with one common exponent
// per CTA (block floating point):
//   - pass A finds the largest exponent of its row group's inputs and converts
//     them to integers below 2^59 (the fields stay FP64 in memory);
//   - every stage records the largest magnitude it wrote (a maximum over the
//     CTA, published by the barrier the stage needs anyway) and the next stage
//     shifts its inputs right, rounding, just far enough that its products stay
//     within their factors' range.  A value is therefore rounded 58 bits or more
//     below the largest one of its CTA's rows or columns (which the other passes
//     add up with it anyway), against FP64's 53 below itself, and additions are
//     exact;
//   - twiddle factors have 62 bits (two limbs); a product is three
//     32 x 32 -> 64 bit multiply-adds per real factor;
//   - W holds the integers; one exponent per row group (pass A) or per CTA of
//     columns (pass B) goes to a small array beside it.  Pass B aligns its
//     column's rows, and pass C its row group's columns, to the largest.
//   - the spectrum multiply keeps the spectrum's own exponents and renormalises
//     by the largest product, so steep spectra lose nothing.
// Against extended-precision transforms the error is 0.3 to 0.6 times the FP64
// butterflies' for k >= 0 and 0.4 to 0.8 times for k < 0 (contact pressures, 64 to
// 2048 a side; 1.7e-16 against 2.9e-16 of the field at 2048 x 2048, k = -0.5).  With
// products of factors below 2^61 and one bit less everywhere (two before inverse
// stages), at the same speed, it was up to 1.3 times theirs for k < 0.  NaN and infinity in an input mark the exponent, which poisons
// the outputs that depend on it (all rows, as an FP64 FFT would) with NaN.
//
// Bound by the integer pipes: about 400 instructions per radix-8 butterfly and
// stage, two thirds of them twiddle products.  Measured (GB300) against FP64
// butterflies: the transform of a 1501 x 1100 grid 1,617 -> 400 us, of 64 x 64
// 57 -> 38 us; there is no size at which FP64 butterflies are faster, so the CG
// and plain modes have no FP64 kernels (the spectrum's set-up, whose result is
// kept in FP64, does).
#pragma once
#include "conv_kernels.cuh"

namespace bem {

using ll = long long;
using fx2 = longlong2;  // a complex value: real and imaginary 64-bit integers

// Products take factors below 2^62 - 2^30 (fsplit).  Components may hold
//   before a forward stage (butterfly, then twiddles)   110e6 2^32 = 2^58.71: the
//     butterfly's values are below (4 + 4 sqrt 2) of that, 2^62 - 2^55; stored 2^62.3
//   before an inverse stage (twiddles, then butterfly)  2^59 - 2^32: its factors
//     1/sqrt 2 meet 8 of that, 2^62 - 2^35; stored below 8 sqrt 2 2^59 = 2^62.5
//   before a leading stage half of whose inputs are zero  2^59: (2 + 2 sqrt 2) of it
//   in W, and before pass C's split (sums of two, one of them multiplied)  2^60
//   before the inverse stage after the spectrum            2^58 (whole bits, rounded up)
// and every bit counts: a value is rounded at its CTA's common exponent, which on a
// steep spectrum is far above most bins.
constexpr int kFxBitsProd = 58, kFxBitsHalf = 59, kFxBitsW = 60;
constexpr unsigned kFxLimitFwd = 110000000u, kFxLimitInv = (1u << 27) - 1;  // high words
constexpr int kFxPoison = 1 << 20;      // exponent of a group that met NaN or infinity
constexpr int kFxZero = -(1 << 20);     // exponent of a group of zeros

__device__ __forceinline__ fx2 fmk(ll x, ll y) { fx2 r; r.x = x; r.y = y; return r; }
__device__ __forceinline__ fx2 fadd(fx2 a, fx2 b) { return fmk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ fx2 fsub(fx2 a, fx2 b) { return fmk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ fx2 fconj(fx2 a) { return fmk(a.x, -a.y); }
// a +- (S i) d
template <int S> __device__ __forceinline__ fx2 fadd_si(fx2 a, fx2 d) {
  return S > 0 ? fmk(a.x - d.y, a.y + d.x) : fmk(a.x + d.y, a.y - d.x);
}
template <int S> __device__ __forceinline__ fx2 fsub_si(fx2 a, fx2 d) { return fadd_si<-S>(a, d); }

__device__ __forceinline__ ll madw(int a, int b, ll c) {
  ll r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// v = h 2^31 + l with l in [-2^30, 2^30), |v| < 2^62 - 2^30
__device__ __forceinline__ void fsplit(ll v, int& h, int& l) {
  const int lo = (int)v, hi = (int)(v >> 32);
  l = (lo << 1) >> 1;
  h = (int)__funnelshift_l((unsigned)lo, (unsigned)hi, 1) + ((lo >> 30) & 1);
}
constexpr ll kFxHalf = 1ll << 30;
// v w, w = (wh 2^31 + wl) / 2^62 with |w| <= 1 (the dropped low product is below one unit)
__device__ __forceinline__ ll frmul(ll v, int wh, int wl) {
  int h, l;
  fsplit(v, h, l);
  const ll mid = madw(l, wh, madw(h, wl, kFxHalf));
  return madw(h, wh, mid >> 31);
}
// Complex product with w (limbs {re h, re l, im h, im l}), or with conj w.  The four
// middle products stay below 2^63: a low limb is below 2^30 but where its component
// is within 2^-31 of 1 (2^31 then), and a butterfly's value with one component near
// 2^62 has the other below 0.61 2^62.
template <bool CONJ>
__device__ __forceinline__ fx2 fcmul(fx2 v, int4 w) {
  int xh, xl, yh, yl;
  fsplit(v.x, xh, xl);
  fsplit(v.y, yh, yl);
  const int ph = CONJ ? -w.z : w.z, pl = CONJ ? -w.w : w.w;  // imaginary limbs
  const int nh = CONJ ? w.z : -w.z, nl = CONJ ? w.w : -w.w;  // and their negatives
  const ll mr = madw(yl, nh, madw(yh, nl, madw(xl, w.x, madw(xh, w.y, kFxHalf))));
  const ll mi = madw(yl, w.x, madw(yh, w.y, madw(xl, ph, madw(xh, pl, kFxHalf))));
  return fmk(madw(yh, nh, madw(xh, w.x, mr >> 31)), madw(yh, w.x, madw(xh, ph, mi >> 31)));
}
// Right shift, rounding to nearest even, s >= 0 (0 for s > 62).  The shifts are
// a few bits, so ties are common, and a tie that always rounds up would bias
// every value alike: the zero frequency then collects it coherently.
__device__ __forceinline__ ll frsh(ll v, int s) {
  if (s <= 0) return v;
  if (s > 62) return 0;
  return (v + ((1ll << (s - 1)) - 1) + ((v >> s) & 1)) >> s;
}
// v 2^-d, rounded; d may be negative (the caller keeps the result in range)
__device__ __forceinline__ ll falign(ll v, int d) {
  if (d >= 0) return frsh(v, d);
  return d < -62 ? 0 : v << -d;
}
// Magnitude word of a component: its bits above the sign, high half.
__device__ __forceinline__ unsigned fmag(ll v) {
  const int hi = (int)(v >> 32);
  return (unsigned)(hi ^ (hi >> 31));
}
__device__ __forceinline__ unsigned fmag(fx2 v) { return max(fmag(v.x), fmag(v.y)); }
// Components are below 2^fbits(mag)
__device__ __forceinline__ int fbits(unsigned mag) { return 64 - __clz((int)mag); }
// Shift that brings high words below LIMIT
template <unsigned LIMIT>
__device__ __forceinline__ int fshift(unsigned mag) {
  if (mag < LIMIT) return 0;
  const int s = 5 - __clz((int)mag);  // mag >> s has 27 bits, as LIMIT
  return (mag >> s) < LIMIT ? s : s + 1;
}

// Maximum over the CTA into a shared word, one atomic per warp; published by the
// caller's next barrier.
__device__ __forceinline__ void cta_max(unsigned* w, unsigned v) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && v) atomicMax(w, v);
}
__device__ __forceinline__ void cta_max(int* w, int v) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) atomicMax(w, v);
}

template <int S> __device__ __forceinline__ void fdft4(fx2& v0, fx2& v1, fx2& v2, fx2& v3) {
  const fx2 a0 = fadd(v0, v2), a1 = fsub(v0, v2), a2 = fadd(v1, v3), d = fsub(v1, v3);
  v0 = fadd(a0, a2); v2 = fsub(a0, a2);
  v1 = fadd_si<S>(a1, d); v3 = fsub_si<S>(a1, d);
}
constexpr int kR2h = 1518500250, kR2l = -25716447;  // 2^62 / sqrt 2 = kR2h 2^31 + kR2l, rounded
__device__ __forceinline__ ll frmul_r2(ll v) { return frmul(v, kR2h, kR2l); }
template <int S> __device__ __forceinline__ void fdft8(fx2* v) {
  fx2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  fx2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  fdft4<S>(e0, e1, e2, e3);
  fdft4<S>(o0, o1, o2, o3);
  // w8 o1 = r (o1.x - S o1.y, o1.y + S o1.x); w8^3 o3 = -r (o3.x + S o3.y, o3.y - S o3.x)
  const fx2 u1 = fmk(frmul_r2(S > 0 ? o1.x - o1.y : o1.x + o1.y), frmul_r2(S > 0 ? o1.y + o1.x : o1.y - o1.x));
  const fx2 u3 = fmk(frmul_r2(S > 0 ? o3.x + o3.y : o3.x - o3.y), frmul_r2(S > 0 ? o3.y - o3.x : o3.y + o3.x));
  v[0] = fadd(e0, o0); v[4] = fsub(e0, o0);
  v[1] = fadd(e1, u1); v[5] = fsub(e1, u1);
  v[2] = fadd_si<S>(e2, o2); v[6] = fsub_si<S>(e2, o2);
  v[3] = fsub(e3, u3); v[7] = fadd(e3, u3);
}

// The stages of a length-2^LOGL transform: the structure, tables' layout and
// shared-memory positions of FftC<double, LOGL>, on integers.
template <int LOGL>
struct FxFft {
  using F = FftC<double, LOGL>;
  static constexpr int L = F::L, L8 = F::L8, R0 = F::R0;
  static __device__ __forceinline__ void stage0_fwd(fx2* v, int t, const int4* tw) {
    if (R0 == 0) {
      fdft8<-1>(v);
#pragma unroll
      for (int q = 1; q < 8; ++q) v[q] = fcmul<false>(v[q], __ldg(tw + t + (q - 1) * L8));
    } else if (R0 == 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        fx2* u = v + 4 * i;
        fdft4<-1>(u[0], u[1], u[2], u[3]);
        const int4* pw = tw + t + i * L8;
#pragma unroll
        for (int q = 1; q < 4; ++q) u[q] = fcmul<false>(u[q], __ldg(pw + (q - 1) * (L >> 2)));
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fx2* u = v + 2 * i;
        const fx2 d = fsub(u[0], u[1]);
        u[0] = fadd(u[0], u[1]);
        u[1] = fcmul<false>(d, __ldg(tw + t + i * L8));
      }
    }
  }
  static __device__ __forceinline__ void stage0_inv(fx2* v, int t, const int4* tw) {
    if (R0 == 0) {
#pragma unroll
      for (int q = 1; q < 8; ++q) v[q] = fcmul<true>(v[q], __ldg(tw + t + (q - 1) * L8));
      fdft8<1>(v);
    } else if (R0 == 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        fx2* u = v + 4 * i;
        const int4* pw = tw + t + i * L8;
#pragma unroll
        for (int q = 1; q < 4; ++q) u[q] = fcmul<true>(u[q], __ldg(pw + (q - 1) * (L >> 2)));
        fdft4<1>(u[0], u[1], u[2], u[3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fx2* u = v + 2 * i;
        const fx2 d = fcmul<true>(u[1], __ldg(tw + t + i * L8));
        u[1] = fsub(u[0], d);
        u[0] = fadd(u[0], d);
      }
    }
  }
  // Radix-8 stages in shared memory, inputs shifted right by s; return the
  // magnitude word of what was written.
  template <bool FWD>
  static __device__ __forceinline__ unsigned stage(fx2* buf, int t, int ls, const int4* tw, int s) {
    const int o = t & ((1 << ls) - 1);
    const int sb = F::sw(((t >> ls) << (ls + 3)) + o);
    fx2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = buf[sb ^ F::sw(r << ls)];
    if (s > 0) {
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = fmk(frsh(v[r].x, s), frsh(v[r].y, s));
    }
    const int4* pw = tw + F::pow_off(ls) + o;
    if (FWD) {
      fdft8<-1>(v);
      if (ls > 0) {
#pragma unroll
        for (int q = 1; q < 8; ++q) v[q] = fcmul<false>(v[q], __ldg(pw + ((q - 1) << ls)));
      }
    } else {
      if (ls > 0) {
#pragma unroll
        for (int q = 1; q < 8; ++q) v[q] = fcmul<true>(v[q], __ldg(pw + ((q - 1) << ls)));
      }
      fdft8<1>(v);
    }
    unsigned m = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      buf[sb ^ F::sw(q << ls)] = v[q];
      m = max(m, fmag(v[q]));
    }
    return m;
  }
};

// Exponent word of an FP64 value: biased exponent, 0 for zero.
__device__ __forceinline__ int dexp(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return (hi | __double2loint(x)) == 0 ? 0 : max(hi >> 20, 1);
}
// x as an integer below 2^kFxBitsHalf in magnitude where the largest biased
// exponent around is emax: x = result * 2^(emax - 1022 - kFxBitsHalf).
__device__ __forceinline__ ll dfix(double x, int emax) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  const ll m = ((ll)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(x);
  const ll q = falign(m, (emax - max(e, 1)) - (kFxBitsHalf - 53));
  return hi < 0 ? -q : q;
}

// Threads per CTA of these kernels are capped as the plan caps them; registers
// for eight complex integers and a product in flight (128).  Row passes of 2048
// and 4096 points, whose CTAs have 512 threads, fit an SM twice at 64 registers:
// they spill about as much as they hold, but one CTA's barriers, loads and
// FP64 conversions are covered by the other's (transform of 2048 x 2048 555 -> 480
// us, 4096 x 1000 529 -> 463, 1501 x 1100 423 -> 390).  Shorter rows, of which
// several CTAs fit anyway, and the column pass only lose by the spills (200 x 251
// 41 -> 47 us; the 4096-point column pass 3% either way by grid).
#define BEM_FX_BOUNDS(LOGL) __launch_bounds__((LOGL) >= 13 ? 1024 : 512, 1)
#define BEM_FX_ROW_BOUNDS(LOGL) __launch_bounds__((LOGL) >= 13 ? 1024 : 512, (LOGL) == 11 || (LOGL) == 12 ? 2 : 1)
constexpr int kFxStages = 8;  // shared magnitude words

// ---------------------------------------------------------------------------
// Pass A: prologue in FP64 (the modes of k_pass_a), one row group per CTA.
template <int MODE, int LOGL>
__device__ __forceinline__ void fx_pass_a_body(const PassArgs<double>& a) {
  using X = FxFft<LOGL>;
  using F = typename X::F;
  constexpr int L8 = F::L8, M = F::L;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double red[3 * 32];
  __shared__ unsigned mag[kFxStages];
  __shared__ int emx;
  fx2* sm = reinterpret_cast<fx2*>(smem_raw);
  Scalars* sc = a.sc;
  if (MODE != A_PLAIN) {
    if (sc->done) return;
  }
  const int nb = a.pl.nbA, lognb = a.pl.lognbA, rs = a.pl.gA.rs;
  const int tid = threadIdx.x;
  const int b = tid >> (LOGL - 3), t = tid & (L8 - 1);
  const int ncols = a.ncols_in, nrows = a.nrows_in, half = (ncols + 1) >> 1;
  int g = blockIdx.x;
  if (MODE == A_CG_T && a.use_band) {  // the contact band's row groups only
    g += sc->band0 / nb;
    if (g * nb > sc->band1) return;
  }
  if (MODE == A_PLAIN && a.use_band == 2) {
    g += a.band_lo / nb;
    if (g * nb > a.band_hi) return;
  }
  const int row0 = g * nb, row = row0 + b;
  if (row0 >= nrows) return;
  const bool act = row < nrows;
  const size_t rowoff = (size_t)row * ncols;
  fx2* buf = sm + b * rs;
  const int4* tw = a.fxA;
  if (tid < kFxStages) mag[tid] = 0;
  if (tid == 0) emx = 0;
  double acc[3] = {0, 0, 0};
  bool upd = false;
  double tau = 0, beta = 0;
  if (MODE == A_PK_P || MODE == A_CG_T) { upd = sc->have_tau != 0; tau = sc->tau; }
  if (MODE == A_PK_T || MODE == A_CG_T) beta = sc->beta;
  if (MODE == A_PK_P && blockIdx.x == 0 && tid == 0) sc->nA = gridDim.x;

  double x[8][2];
  {
    PIn<double> in[8][2] = {};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!F::first_half(e)) continue;
      const int n = F::n0(t, e);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (act && n < half && 2 * n + h < ncols) pro_gather<double, MODE>(a, rowoff + 2 * n + h, in[e][h]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!F::first_half(e)) continue;
      const int n = F::n0(t, e);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        x[e][h] = 0.0;
        if (act && n < half && 2 * n + h < ncols)
          x[e][h] = pro_apply<double, MODE>(a, rowoff + 2 * n + h, in[e][h], upd, tau, beta, acc);
      }
    }
  }
  int em = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (!F::first_half(e)) continue;
    em = max(em, max(dexp(x[e][0]), dexp(x[e][1])));
  }
  __syncthreads();
  cta_max(&emx, em);
  __syncthreads();
  const int emax = emx;
  fx2 v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    v[e] = fmk(0, 0);
    if (!F::first_half(e)) continue;
    if (emax > 0 && emax < 0x7ff) v[e] = fmk(dfix(x[e][0], emax), dfix(x[e][1], emax));
  }
  int ex = emax == 0 ? kFxZero : emax == 0x7ff ? kFxPoison : emax - 1022 - kFxBitsHalf;
  X::stage0_fwd(v, t, tw);
  unsigned m = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    buf[F::ix0(t, e)] = v[e];
    m = max(m, fmag(v[e]));
  }
  cta_max(&mag[0], m);
  __syncthreads();
  int st = 0;
#pragma unroll
  for (int ls = F::LS_TOP; ls >= 0; ls -= 3) {
    const int s = fshift<kFxLimitFwd>(mag[st]);
    ex += s;
    m = X::template stage<true>(buf, t, ls, tw, s);
    cta_max(&mag[++st], m);
    __syncthreads();
  }
  const int s = max(0, fbits(mag[st]) - kFxBitsW);
  ex += s;
  if (MODE == A_PK_P) block_partials<double, 3>(acc, a.partA + 4 * blockIdx.x, red);
  // X[k] = (z[k] + conj z[M-k])/2 + w_k (z[k] - conj z[M-k])/(2i), twice that here:
  // the group's exponent takes the factor 1/2
  if (tid == 0) a.fx_ea[g] = ex <= kFxZero / 2 ? kFxZero : ex >= kFxPoison / 2 ? kFxPoison : ex - 1;
  constexpr int hm = M / 2 + 1;
  const int rows = min(nb, nrows - row0), rows_w = a.rows_w;
  fx2* W = reinterpret_cast<fx2*>(a.W);
  const int* sp = a.spA;
  for (int idx = tid; idx < hm << lognb; idx += blockDim.x) {
    const int k = idx >> lognb, bb = idx & (nb - 1);
    if (bb >= rows) continue;
    const fx2* z = sm + bb * rs;
    fx2 xk, xm;
    if (k == 0) {
      const fx2 z0 = z[0];
      const ll p = frsh(z0.x, s), q = frsh(z0.y, s);
      xk = fmk(2 * (p + q), 0);
      xm = fmk(2 * (p - q), 0);
    } else {
      fx2 c = z[__ldg(sp + k)], d = z[__ldg(sp + M - k)];
      c = fmk(frsh(c.x, s), frsh(c.y, s));
      d = fmk(frsh(d.x, s), frsh(d.y, s));
      const fx2 E = fmk(c.x + d.x, c.y - d.y);        // c + conj d
      const fx2 O = fmk(c.y + d.y, d.x - c.x);        // (c - conj d) / i
      const fx2 wO = fcmul<false>(O, __ldg(a.fxS + k));
      xk = fadd(E, wO);
      xm = fconj(fsub(E, wO));                         // X[M-k] = conj(E - w O)
    }
    const int km = k == 0 ? M : M - k;
    if (!bem_check((size_t)km * rows_w + row0 + bb < (size_t)(M + 1) * rows_w && row0 + bb < rows_w, a.kerr)) continue;
    W[(size_t)k * rows_w + row0 + bb] = xk;
    if (km != k) W[(size_t)km * rows_w + row0 + bb] = xm;
  }
}

// ---------------------------------------------------------------------------
// Pass B: column FFT, spectrum multiply, inverse; nbB columns per CTA.
template <int LOGL>
__device__ __forceinline__ void fx_pass_b_body(const PassArgs<double>& a) {
  using X = FxFft<LOGL>;
  using F = typename X::F;
  constexpr int L = F::L, L8 = F::L8, hyq = (L >> 1) + 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ unsigned mag[2 * kFxStages];
  __shared__ int emx[2];
  fx2* sm = reinterpret_cast<fx2*>(smem_raw);
  if (a.sc != nullptr && a.sc->done) return;
  const int M = a.pl.M, rin = a.rows_w, rs = a.pl.gB.rs, lognbA = a.pl.lognbA;
  const int tid = threadIdx.x;
  const int c = tid >> (LOGL - 3), t = tid & (L8 - 1);
  const int kx = blockIdx.x * a.pl.nbB + c;
  const bool act = kx <= M;
  fx2* buf = sm + c * rs;
  const int4* tw = a.fxB;
  const int* sp = a.spB;
  fx2* W = reinterpret_cast<fx2*>(a.W);
  const size_t coff = (size_t)(act ? kx : 0) * rin;
  int ylo = 0, yhi = rin - 1;
  if (a.use_band) {
    ylo = a.use_band == 2 ? a.band_lo : a.sc->band0;
    yhi = min(a.use_band == 2 ? a.band_hi : a.sc->band1, rin - 1);
  }
  if (tid < 2 * kFxStages) mag[tid] = 0;
  if (tid < 2) emx[tid] = kFxZero;

  fx2 v[8];
  int ev[8];
  int em = kFxZero;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    v[e] = fmk(0, 0);
    ev[e] = kFxZero;
    if (!F::first_half(e)) continue;
    const int y = F::n0(t, e);
    if (act && y >= ylo && y <= yhi && bem_check(coff + y < (size_t)(M + 1) * rin, a.kerr)) {
      v[e] = W[coff + y];
      ev[e] = __ldg(a.fx_ea + (y >> lognbA));
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (!F::first_half(e)) continue;
    if (ev[e] > kFxZero / 2) em = max(em, ev[e] + fbits(fmag(v[e])));
  }
  __syncthreads();
  cta_max(&emx[0], em);
  __syncthreads();
  int ex = emx[0] - kFxBitsHalf;
  const bool poison = emx[0] >= kFxPoison / 2, zero = emx[0] <= kFxZero / 2;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (!F::first_half(e)) continue;
    const int d = ex - ev[e];
    if (poison || ev[e] <= kFxZero / 2) v[e] = fmk(0, 0);
    else v[e] = fmk(falign(v[e].x, d), falign(v[e].y, d));
  }
  X::stage0_fwd(v, t, tw);
  unsigned m = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    buf[F::ix0(t, e)] = v[e];
    m = max(m, fmag(v[e]));
  }
  cta_max(&mag[0], m);
  __syncthreads();
  int st = 0;
#pragma unroll
  for (int ls = F::LS_TOP; ls >= 3; ls -= 3) {
    const int s = fshift<kFxLimitFwd>(mag[st]);
    ex += s;
    m = X::template stage<true>(buf, t, ls, tw, s);
    cta_max(&mag[++st], m);
    __syncthreads();
  }
  // stride-1 stage, spectrum multiply, first inverse stage in registers: thread
  // t holds the frequencies t + q L/8.  The products keep their factors'
  // exponents until the largest is known.
  {
    const int sp0 = __ldg(sp + t);
    const double* kc = a.khat + (size_t)(act ? kx : 0) * hyq;
    double kf[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int ky = t + q * L8;
      const int kk = ky <= (L >> 1) ? ky : L - ky;
      kf[q] = act ? __ldg(kc + kk) : 0.0;
    }
    const int s = fshift<kFxLimitFwd>(mag[st]);
    ex += s;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = buf[sp0 ^ r];
      if (s > 0) v[r] = fmk(frsh(v[r].x, s), frsh(v[r].y, s));
    }
    fdft8<-1>(v);
    em = kFxZero;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      // kf = +- (h 2^31 + l) 2^(ek - 62), h 2^31 + l in [2^61, 2^62)
      const int hi = __double2hiint(kf[q]), e = (hi >> 20) & 0x7ff;
      const ll mm = (((ll)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(kf[q])) << 9;
      const int h = (int)(mm >> 31), l = (int)(mm & 0x7fffffff);
      fx2 y = fmk(frmul(v[q].x, h, l), frmul(v[q].y, h, l));
      if (hi < 0) y = fmk(-y.x, -y.y);
      v[q] = y;
      ev[q] = e == 0x7ff ? kFxPoison : max(e, 1) - 1022;
      if (mm != 0) em = max(em, ev[q] + fbits(fmag(y)));
    }
    cta_max(&emx[1], em);
    __syncthreads();
    const int e1 = emx[1] - kFxBitsProd;  // exponent of the aligned products, on top of ex
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int d = e1 - ev[q];
      v[q] = d > 62 || d < -62 ? fmk(0, 0) : fmk(falign(v[q].x, d), falign(v[q].y, d));
    }
    ex += emx[1] > kFxZero / 2 ? e1 : 0;
    fdft8<1>(v);
    m = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      buf[sp0 ^ r] = v[r];
      m = max(m, fmag(v[r]));
    }
    cta_max(&mag[++st], m);
  }
  __syncthreads();
#pragma unroll
  for (int ls = 3; ls <= F::LS_TOP; ls += 3) {
    const int s = fshift<kFxLimitInv>(mag[st]);
    ex += s;
    m = X::template stage<false>(buf, t, ls, tw, s);
    cta_max(&mag[++st], m);
    __syncthreads();
  }
  const int s = fshift<kFxLimitInv>(mag[st]);
  ex += s;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    v[e] = buf[F::ix0(t, e)];
    if (s > 0) v[e] = fmk(frsh(v[e].x, s), frsh(v[e].y, s));
  }
  X::stage0_inv(v, t, tw);
  if (act) {
    if (t == 0) a.fx_eb[kx] = poison || emx[1] >= kFxPoison / 2 ? kFxPoison : zero ? kFxZero : ex;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!F::first_half(e)) continue;
      const int y = F::n0(t, e);
      if (y >= ylo && y <= yhi && bem_check(coff + y < (size_t)(M + 1) * rin, a.kerr)) W[coff + y] = v[e];
    }
  }
}

// ---------------------------------------------------------------------------
// Pass C: inverse rows, epilogue in FP64 (the modes of k_pass_c).
template <int MODE, int LOGL>
__device__ __forceinline__ void fx_pass_c_body(const PassArgs<double>& a) {
  using X = FxFft<LOGL>;
  using F = typename X::F;
  constexpr int L8 = F::L8, M = F::L;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double red[4 * 32];
  __shared__ int lastflag;
  __shared__ unsigned mag[kFxStages];
  __shared__ int emx;
  __shared__ CgPre pre;
  fx2* sm = reinterpret_cast<fx2*>(smem_raw);
  Scalars* sc = a.sc;
  if (MODE != C_PLAIN && MODE != C_GAP) {
    if (sc->done) return;
  }
  if (MODE == C_CG_R) cg_pre_load(sc, &pre);
  const int nb = a.pl.nbA, lognb = a.pl.lognbA, rs = a.pl.gA.rs;
  const int nx = a.pl.nx, ny = a.pl.ny;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int b = tid >> (LOGL - 3), t = tid & (L8 - 1);
  // row groups g0 .. g0+ng-1; an empty band keeps one CTA for the scalar work
  // (rows of an edge group outside the band hold no transform: read as zero)
  int g0 = 0, ng = (ny + nb - 1) / nb, rlo = 0, rhi = ny - 1;
  if (MODE == C_CG_R && a.use_band) {
    rlo = sc->band0;
    rhi = min(sc->band1, ny - 1);
    g0 = rlo / nb;
    ng = rhi >= rlo ? rhi / nb + 1 - g0 : 0;
  }
  if (MODE == C_GAP && a.use_band == 2) {
    rlo = a.band_lo;
    rhi = min(a.band_hi, ny - 1);
    g0 = rlo / nb;
    ng = rhi >= rlo ? rhi / nb + 1 - g0 : 0;
  }
  const int g = g0 + blockIdx.x;
  if ((int)blockIdx.x >= max(ng, 1)) return;
  double acc[4] = {0, 0, 0, 0};
  if (ng > 0) {
    const int row0 = g * nb;
    const fx2* W = reinterpret_cast<const fx2*>(a.W);
    const int4* tw = a.fxA;
      const int* sp = a.spA;
    if (tid < kFxStages) mag[tid] = 0;
    if (tid == 0) emx = kFxZero;
    constexpr int hm = (M >> 1) + 1;
    const int total = hm << lognb;
    constexpr int NP = 5;  // ceil((M/2 + 1) nb / (nb M/8)) for M >= 16
    fx2 xk[NP], xm[NP];
    int ek[NP], ej[NP];
    int em = kFxZero;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int idx = tid + j * nthr;
      xk[j] = fmk(0, 0);
      xm[j] = fmk(0, 0);
      ek[j] = ej[j] = kFxZero;
      if (idx < total) {
        const int k = idx >> lognb, rw = row0 + (idx & (nb - 1));
        ek[j] = __ldg(a.fx_eb + k);
        ej[j] = __ldg(a.fx_eb + M - k);
        if (rw >= rlo && rw <= rhi && bem_check(k <= M && rw < a.rows_w, a.kerr)) {
          xk[j] = W[(size_t)k * a.rows_w + rw];
          xm[j] = W[(size_t)(M - k) * a.rows_w + rw];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      if (ek[j] > kFxZero / 2) em = max(em, ek[j] + fbits(fmag(xk[j])));
      if (ej[j] > kFxZero / 2) em = max(em, ej[j] + fbits(fmag(xm[j])));
    }
    __syncthreads();
    cta_max(&emx, em);
    __syncthreads();
    const int e0 = emx;
    const bool poison = e0 >= kFxPoison / 2, zero = e0 <= kFxZero / 2;
    int ex = e0 - kFxBitsW;
    unsigned m = 0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int idx = tid + j * nthr;
      if (idx >= total) continue;
      const int k = idx >> lognb, bb = idx & (nb - 1);
      fx2* z = sm + bb * rs;
      fx2 p = xk[j], q = xm[j];
      const int dk = ex - ek[j], dj = ex - ej[j];
      p = poison || ek[j] <= kFxZero / 2 ? fmk(0, 0) : fmk(falign(p.x, dk), falign(p.y, dk));
      q = poison || ej[j] <= kFxZero / 2 ? fmk(0, 0) : fmk(falign(q.x, dj), falign(q.y, dj));
      // Z[k] = E + i O e^{+i pi k/M}, E = X[k] + conj X[M-k], O = X[k] - conj X[M-k]
      const fx2 E = fmk(p.x + q.x, p.y - q.y);
      const fx2 O = fcmul<true>(fmk(p.x - q.x, p.y + q.y), __ldg(a.fxS + k));
      const fx2 zk = fmk(E.x - O.y, E.y + O.x);
      z[__ldg(sp + k)] = zk;
      m = max(m, fmag(zk));
      if (k != 0 && k != M - k) {
        const fx2 zm = fmk(E.x + O.y, O.x - E.y);  // conj(E - i O)
        z[__ldg(sp + M - k)] = zm;
        m = max(m, fmag(zm));
      }
    }
    cta_max(&mag[0], m);
    __syncthreads();
    fx2* buf = sm + b * rs;
    int st = 0;
#pragma unroll
    for (int ls = 0; ls <= F::LS_TOP; ls += 3) {
      const int s = fshift<kFxLimitInv>(mag[st]);
      ex += s;
      m = X::template stage<false>(buf, t, ls, tw, s);
      cta_max(&mag[++st], m);
      __syncthreads();
    }
    const int row = row0 + b;
    const bool act = row < ny;
    const size_t rowoff = (size_t)row * nx;
    const int half = (nx + 1) >> 1;
    EIn<double> ein[8][2] = {};
    if (MODE != C_PLAIN) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (!F::first_half(e)) continue;
        const int n = F::n0(t, e);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (act && n < half && 2 * n + h < nx) epi_gather<double, MODE>(a, rowoff + 2 * n + h, ein[e][h]);
      }
    }
    const int s = fshift<kFxLimitInv>(mag[st]);
    ex += s;
    fx2 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      v[e] = buf[F::ix0(t, e)];
      if (s > 0) v[e] = fmk(frsh(v[e].x, s), frsh(v[e].y, s));
    }
    X::stage0_inv(v, t, tw);
    // far from 1 the factor alone could leave FP64's range where the product does not
    const bool wide = ex < -900 || ex > 900;
    const double us = poison ? __longlong_as_double(0x7ff8000000000000ll)
                             : zero ? 0.0 : wide ? a.uscale : scalbn(a.uscale, ex);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!F::first_half(e)) continue;
      const int n = F::n0(t, e);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (act && n < half && 2 * n + h < nx) {
          double u = us * (double)(h ? v[e].y : v[e].x);
          if (wide && !poison && !zero) u = scalbn(u, ex);
          epi_apply<double, MODE>(a, rowoff + 2 * n + h, u, ein[e][h], acc);
        }
    }
  } else if (MODE == C_PLAIN || MODE == C_GAP) {
    return;
  }
  if (MODE == C_PLAIN || MODE == C_GAP) return;
  constexpr int NQ = MODE == C_CG_R ? 4 : 2;
  const int ncta = max(ng, 1);
  block_partials<double, NQ>(acc, a.partC + 4 * blockIdx.x, red);
  if (!last_block_arrival_of(MODE == C_PK_G ? &sc->cnt_c : &sc->cnt_a, &lastflag, ncta)) return;
  double s2[4] = {0, 0, 0, 0};
  grid_sum<double, NQ>(a.partC, ncta, s2, red);
  double s3[3] = {0, 0, 0};
  if (MODE == C_PK_G) grid_sum<double, 3>(a.partA, __ldcg(&sc->nA), s3, red);
  if (tid != 0) return;
  pass_c_finalize<double, MODE>(sc, s2, s3, pre);
}

template <int MODE, int LOGL>
__global__ void BEM_FX_ROW_BOUNDS(LOGL) k_fx_a(PassArgs<double> a) { fx_pass_a_body<MODE, LOGL>(a); }
template <int MODE, int LOGL>
__global__ void BEM_FX_ROW_BOUNDS(LOGL) k_fx_a_mi(const PassArgs<double>* __restrict__ arr) {
  fx_pass_a_body<MODE, LOGL>(arr[blockIdx.y]);
}
template <int LOGL>
__global__ void BEM_FX_BOUNDS(LOGL) k_fx_b(PassArgs<double> a) { fx_pass_b_body<LOGL>(a); }
template <int LOGL>
__global__ void BEM_FX_BOUNDS(LOGL) k_fx_b_mi(const PassArgs<double>* __restrict__ arr) {
  fx_pass_b_body<LOGL>(arr[blockIdx.y]);
}
template <int MODE, int LOGL>
__global__ void BEM_FX_ROW_BOUNDS(LOGL) k_fx_c(PassArgs<double> a) { fx_pass_c_body<MODE, LOGL>(a); }
template <int MODE, int LOGL>
__global__ void BEM_FX_ROW_BOUNDS(LOGL) k_fx_c_mi(const PassArgs<double>* __restrict__ arr) {
  fx_pass_c_body<MODE, LOGL>(arr[blockIdx.y]);
}

// ---------------------------------------------------------------------------
// Host launchers: one row group (or nbB columns) per CTA.
template <int MODE>
void launch_fx_a_mode(const PassArgs<double>& a, const PassArgs<double>* arr, int n, cudaStream_t s) {
  const dim3 grid((a.nrows_in + a.pl.nbA - 1) / a.pl.nbA, n), block(a.pl.threadsA);
  switch (a.pl.gA.logL) {
#define BEM_CASE(LG)                                                              \
  case LG:                                                                        \
    if (arr) {                                                                    \
      if constexpr (MODE != A_PLAIN) k_fx_a_mi<MODE, LG><<<grid, block, a.pl.smemA, s>>>(arr); \
    } else {                                                                      \
      k_fx_a<MODE, LG><<<grid, block, a.pl.smemA, s>>>(a);                        \
    }                                                                             \
    break;
    BEM_LOGL_CASES_A(BEM_CASE)
#undef BEM_CASE
  }
}
template <int MODE>
void launch_fx_c_mode(const PassArgs<double>& a, const PassArgs<double>* arr, int n, cudaStream_t s) {
  const dim3 grid(a.pl.gridA, n), block(a.pl.threadsA);
  switch (a.pl.gA.logL) {
#define BEM_CASE(LG)                                                              \
  case LG:                                                                        \
    if (arr) {                                                                    \
      if constexpr (MODE == C_PK_G || MODE == C_PK_R || MODE == C_CG_R)           \
        k_fx_c_mi<MODE, LG><<<grid, block, a.pl.smemC, s>>>(arr);                 \
    } else {                                                                      \
      k_fx_c<MODE, LG><<<grid, block, a.pl.smemC, s>>>(a);                        \
    }                                                                             \
    break;
    BEM_LOGL_CASES_A(BEM_CASE)
#undef BEM_CASE
  }
}

}  // namespace bem
