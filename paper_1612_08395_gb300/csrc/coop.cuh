// CG loops of medium grids in one cooperative launch (FP32 path).
//
// On sub-grids of 256 to 1024 elements a side the three passes of a fixed-set
// CG iteration take 36 us on the 2048^2 torus although their instructions need
// about 15: each pass starts cold (launch gap, scalar reads, staging set-up,
// first loads) and ends with one CTA adding everybody's sums.  Here the whole
// loop is one kernel of one CTA per SM:
//   - a CTA owns R grid rows for the whole loop and keeps their p, g, t and r
//     (or c) in shared memory; only W crosses the chip, through L2;
//   - phases are separated by a grid barrier (arrive on a counter, poll it):
//     three per transform;
//   - every CTA adds all CTAs' partial sums itself, in the same order, and takes
//     the scalar decisions from its own copy, so no CTA waits for another's
//     serial tail beyond the barrier.
// Only the rows that can hold pressure (the box of the held or overlap set) are
// transformed.  The arithmetic is that of the passes; the order of the partial
// sums differs.
//
// The CTAs wait for one another, so all must be resident, and another stream's
// long kernel may hold some of them back.  They gather first: if one has waited a
// tenth of a second for the others, all leave, nothing has been written, and the
// host runs the loop as passes, which need no such thing.  Once gathered, no wait
// depends on other work; each is bounded all the same, and a CTA that gives up
// there sets the handle's error word and leaves, and so do the others.
//
// Bound by the barriers and the L2 round trips of W between them.  Measured
// (GB300, per fixed-set iteration; a Polonsky-Keer one takes twice that): 256 x 256
// 11 us (15 in a cluster, 18 as passes), 512 x 512 14 us (21 as passes), 1024 x 1024
// with every row held 29 us (33 as passes); the 401 depths of the 2048 x 2048
// pull-off, on sub-grids of 1024 and 512, 23.1 -> 14.0 s (with the FP64 path's
// integer transforms, about a seventh of that).
#pragma once
#include "resident.cuh"

namespace bem {

template <int LM, int LP>
struct CoopGeo {
  static constexpr int M = 1 << LM, P = 1 << LP, NY = P / 2;
  static constexpr int TR = M / 8, TC = P / 8;
  // four columns a round (2048 points: 1024 threads of 64 registers)
  static constexpr int NT = LP == 11 ? 1024 : LP == 10 || LM == 10 ? 512 : 256;
  static constexpr int RPR = NT / TR < 8 ? NT / TR : 8, CPR = NT / TC < 8 ? NT / TC : 8;  // rows, columns per round
  static constexpr int RS = M + kGeo8[LM - 3].pad[res_lg(RPR)];
  static constexpr int CZ = P + kGeo8[LP - 3].pad[res_lg(CPR)];
  static constexpr int work = (RPR * RS > CPR * CZ ? RPR * RS : CPR * CZ);  // float2
  static constexpr int RMAX = 2 * RPR < 16 ? 2 * RPR : 16;                  // rows per CTA at most
};

// State of the grid barrier and the partial sums (device memory of the handle).
constexpr int kCoopMaxCtas = 256;
struct CoopShared {
  unsigned int count;                    // arrivals at the grid barrier
  unsigned int gathered;                 // 0: CTAs are missing, 1: all are here, 2: given up
  unsigned int pad[30];
  float2 part[2][kCoopMaxCtas * 8];      // alternating between consecutive sums
};

// The gathering: thread 0 of every CTA arrives, and asks after the loads that
// need no other CTA whether all came.  The last to arrive and the first to run out
// of patience both try to settle it; whoever does, all CTAs see the same answer.
constexpr unsigned long long kCoopGatherNs = 100000000ull;
__device__ __forceinline__ void coop_arrive(CoopShared* cs, int nb) {
  if (atomicAdd(&cs->count, 1u) + 1 == (unsigned)nb) atomicCAS(&cs->gathered, 0u, 1u);
}
__device__ __forceinline__ bool coop_all_came(CoopShared* cs) {
  unsigned v;
  unsigned long long t0 = 0;
  for (int i = 0;; ++i) {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&cs->gathered) : "memory");
    if (v) return v == 1;
    if ((i & 1023) == 1023) {
      const unsigned long long t = global_ns();
      if (!t0) t0 = t;
      else if (t - t0 > kCoopGatherNs) {
        const unsigned old = atomicCAS(&cs->gathered, 0u, 2u);
        return old == 1;
      }
    }
  }
}

// Grid barrier: every CTA's earlier global writes are visible to every CTA
// afterwards (read with L2 loads).  One counter, polled by one thread per CTA: a
// word per CTA polled by everybody's first warp keeps the L2 busy with the polls
// (a fixed-set iteration of 129 CTAs took 29 us instead of 14).  False: the wait
// ran out (about a second).
__device__ __forceinline__ bool coop_grid_sync(CoopShared* cs, int nb, unsigned* target, int* bad) {
  *target += nb;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned v;
    asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(&cs->count) : "memory");
    ++v;
    unsigned long long t0 = 0;
    for (int i = 0; (int)(v - *target) < 0; ++i) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&cs->count) : "memory");
      if ((i & 1023) == 1023) {
        const unsigned long long t = global_ns();
        if (!t0) t0 = t;
        else if (t - t0 > kMbarMaxNs) { *bad = 1; break; }
      }
    }
  }
  __syncthreads();
  return *bad == 0;
}

template <int LM, int LP>
struct Coop {
  using Gm = CoopGeo<LM, LP>;
  using FR = FftC<float, LM>;
  using FC = FftC<float, LP>;
  static constexpr int M = Gm::M, P = Gm::P;
  static __device__ __forceinline__ constexpr int slot(int e) {
    return FR::R0 == 0 ? e : FR::R0 == 2 ? (e >> 2) * 2 + (e & 1) : e >> 1;
  }
  template <int N> static __device__ __forceinline__ void group_sync(int g) {
    if (N <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(N) : "memory");
  }

  struct Ctx {
    const PassArgs<float>* a;
    CoopShared* cs;
    float2* work;
    int R, rows, nb, blk;  // rows per CTA, rows in all, CTAs, this CTA
    unsigned target;       // barrier count after the last barrier
    int* bad;              // shared: a wait ran out
    int magic;             // ceil(65536 / (R / 2))
  };

  static __device__ __forceinline__ bool grid_sync(Ctx& c) {
    return coop_grid_sync(c.cs, c.nb, &c.target, c.bad);
  }

  // Rows: transform input x(row slot, element pair index) -> W.
  template <class GetX>
  static __device__ __forceinline__ void phase_a(Ctx& c, GetX&& getx) {
    const PassArgs<float>& a = *c.a;
    const int tid = threadIdx.x, b = tid / Gm::TR, t = tid % Gm::TR;
    const float2* tw = reinterpret_cast<const float2*>(a.twA);
    const float2* tws = reinterpret_cast<const float2*>(a.twS);
    const int* sp = a.spA;
    float2* W = reinterpret_cast<float2*>(a.W);
    for (int r0 = 0; r0 < c.R; r0 += Gm::RPR) {
      const int sl = r0 + b, row = c.blk * c.R + sl;
      const bool ra = b < Gm::RPR && sl < c.R && row < c.rows;  // whole row groups
      if (r0) __syncthreads();  // the previous rows' spectra are stored
      if (ra) {
        float2* buf = c.work + b * Gm::RS;
        float2 v[8];
        getx(sl, t, v);
        FR::stage0_fwd(v, t, tw);
#pragma unroll
        for (int e = 0; e < 8; ++e) buf[FR::ix0(t, e)] = v[e];
        group_sync<Gm::TR>(b);
#pragma unroll
        for (int ls = FR::LS_TOP; ls >= 0; ls -= 3) {
          FR::dif(buf, t, ls, tw);
          group_sync<Gm::TR>(b);
        }
      }
      __syncthreads();
      const int rr = min(Gm::RPR, c.R - r0), rp = rr >> 1;  // even
      const int magic = rr == c.R ? c.magic : (65535 + rp) / rp;
      for (int idx = tid; idx < (M / 2 + 1) * rp; idx += Gm::NT) {
        const int k = (idx * magic) >> 16, bb = 2 * (idx - k * rp);
        const int y = c.blk * c.R + r0 + bb;
        if (y >= c.rows) continue;
        const float2* s0 = c.work + bb * Gm::RS;
        const float2* s1 = s0 + Gm::RS;
        const bool two = y + 1 < c.rows;
        float2 xk0, xm0, xk1 = make_float2(0.f, 0.f), xm1 = make_float2(0.f, 0.f);
        if (k == 0) {
          const float2 z0 = s0[0];
          xk0 = make_float2(z0.x + z0.y, 0.f);
          xm0 = make_float2(z0.x - z0.y, 0.f);
          if (two) {
            const float2 z1 = s1[0];
            xk1 = make_float2(z1.x + z1.y, 0.f);
            xm1 = make_float2(z1.x - z1.y, 0.f);
          }
        } else {
          const int pk = __ldg(sp + k), pm = __ldg(sp + M - k);
          const float2 w = __ldg(tws + k);
          split_two<float>(s0, pk, pm, w, xk0, xm0);
          if (two) split_two<float>(s1, pk, pm, w, xk1, xm1);
        }
        const int km = k == 0 ? M : M - k;
        // rows_w is even: the pair is inside W's row even where y + 1 is past the last row
        if (!bem_check(k <= M && km <= M && y + 1 < a.rows_w, a.kerr)) continue;
        __stcg(reinterpret_cast<float4*>(W + (size_t)k * a.rows_w + y), make_float4(xk0.x, xk0.y, xk1.x, xk1.y));
        if (km != k)
          __stcg(reinterpret_cast<float4*>(W + (size_t)km * a.rows_w + y), make_float4(xm0.x, xm0.y, xm1.x, xm1.y));
      }
    }
  }

  static __device__ __forceinline__ void phase_b(Ctx& c) {
    const PassArgs<float>& a = *c.a;
    constexpr int L = P, L8 = Gm::TC, hyq = L / 2 + 1;
    const int tid = threadIdx.x, cc = tid / Gm::TC, t = tid % Gm::TC;
    const float2* tw = reinterpret_cast<const float2*>(a.twB);
    float2* W = reinterpret_cast<float2*>(a.W);
    float2* cz = c.work + (cc < Gm::CPR ? cc : 0) * Gm::CZ;
    const int k0 = (int)((long long)(M + 1) * c.blk / c.nb), k1 = (int)((long long)(M + 1) * (c.blk + 1) / c.nb);
    const int sp0 = __ldg(a.spB + t);
    for (int kb = k0; kb < k1; kb += Gm::CPR) {
      const int kx = kb + cc;
      if (cc >= Gm::CPR || kx >= k1) {
        if (Gm::TC > 32) continue;  // whole column groups
      }
      float2* w = W + (size_t)kx * a.rows_w;
      float2 v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        v[e] = make_float2(0.f, 0.f);
        if (!FC::first_half(e)) continue;
        const int y = FC::n0(t, e);
        if (y < c.rows && bem_check(kx <= M && y < a.rows_w, a.kerr)) v[e] = __ldcg(w + y);
      }
      FC::stage0_fwd(v, t, tw);
#pragma unroll
      for (int e = 0; e < 8; ++e) cz[FC::ix0(t, e)] = v[e];
      group_sync<Gm::TC>(cc);
#pragma unroll
      for (int ls = FC::LS_TOP; ls >= 3; ls -= 3) {
        FC::dif(cz, t, ls, tw);
        group_sync<Gm::TC>(cc);
      }
      {
        const float* kc = a.khat + (size_t)kx * hyq;
        float kf[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int ky = t + q * L8;
          kf[q] = __ldg(kc + (ky <= (L >> 1) ? ky : L - ky));
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = cz[sp0 ^ r];
        dft8<float, -1>(v);
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = scale<float>(v[q], kf[q]);
        dft8<float, 1>(v);
#pragma unroll
        for (int r = 0; r < 8; ++r) cz[sp0 ^ r] = v[r];
      }
      group_sync<Gm::TC>(cc);
#pragma unroll
      for (int ls = 3; ls <= FC::LS_TOP; ls += 3) {
        FC::dit(cz, t, ls, tw);
        group_sync<Gm::TC>(cc);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = cz[FC::ix0(t, e)];
      FC::stage0_inv(v, t, tw);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (!FC::first_half(e)) continue;
        const int y = FC::n0(t, e);
        if (y < c.rows && bem_check(kx <= M && y < a.rows_w, a.kerr)) __stcg(w + y, v[e]);
      }
    }
  }

  // Rows: W -> the inverse transform's values v (unscaled) of each row slot.
  template <class Put>
  static __device__ __forceinline__ void phase_c(Ctx& c, Put&& put) {
    const PassArgs<float>& a = *c.a;
    const int tid = threadIdx.x, b = tid / Gm::TR, t = tid % Gm::TR;
    const float2* tw = reinterpret_cast<const float2*>(a.twA);
    const float2* tws = reinterpret_cast<const float2*>(a.twS);
    const int* sp = a.spA;
    const float2* W = reinterpret_cast<const float2*>(a.W);
    for (int r0 = 0; r0 < c.R; r0 += Gm::RPR) {
      if (r0) __syncthreads();
      const int rr = min(Gm::RPR, c.R - r0), rp = rr >> 1;
      const int magic = rr == c.R ? c.magic : (65535 + rp) / rp;
#pragma unroll 2
      for (int idx = tid; idx < (M / 2 + 1) * rp; idx += Gm::NT) {
        const int k = (idx * magic) >> 16, bb = 2 * (idx - k * rp);
        const int y = c.blk * c.R + r0 + bb;
        if (y >= c.rows || !bem_check(k <= M && y + 1 < a.rows_w, a.kerr)) continue;
        const float4 fk = __ldcg(reinterpret_cast<const float4*>(W + (size_t)k * a.rows_w + y));
        const float4 fm = __ldcg(reinterpret_cast<const float4*>(W + (size_t)(M - k) * a.rows_w + y));
        const int pk = __ldg(sp + k), pm = k ? __ldg(sp + M - k) : 0;
        const float2 wk = conj<float>(__ldg(tws + k));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float2* s = c.work + (bb + h) * Gm::RS;
          const float2 xk = h ? make_float2(fk.z, fk.w) : make_float2(fk.x, fk.y);
          const float2 xm = h ? make_float2(fm.z, fm.w) : make_float2(fm.x, fm.y);
          const float2 E = add<float>(xk, conj<float>(xm));
          const float2 O = mul<float>(sub<float>(xk, conj<float>(xm)), wk);
          s[pk] = add<float>(E, mul_si<float, 1>(O));
          if (k != 0 && k != M - k) {
            const float2 wm = make_float2(-wk.x, wk.y);
            const float2 E2 = add<float>(xm, conj<float>(xk));
            const float2 O2 = mul<float>(sub<float>(xm, conj<float>(xk)), wm);
            s[pm] = add<float>(E2, mul_si<float, 1>(O2));
          }
        }
      }
      __syncthreads();
      const int sl = r0 + b, row = c.blk * c.R + sl;
      if (b < Gm::RPR && sl < c.R && row < c.rows) {
        float2* buf = c.work + b * Gm::RS;
#pragma unroll
        for (int ls = 0; ls <= FR::LS_TOP; ls += 3) {
          FR::dit(buf, t, ls, tw);
          group_sync<Gm::TR>(b);
        }
        float2 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = buf[FR::ix0(t, e)];
        FR::stage0_inv(v, t, tw);
        put(sl, t, v);
      }
    }
  }

  // Grid sums of NQ per-thread values: the totals (float-float) in every lane of
  // warp 0 of every CTA, the same in all.  Includes a grid barrier.
  template <int NQ>
  static __device__ __forceinline__ bool sum(Ctx& c, const float* acc, float2* red, int* par, float2* v) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int nw = Gm::NT / 32;
    float2* part = c.cs->part[*par];
    *par ^= 1;
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = make_float2(acc[q], 0.f);
    warp_sum_store<NQ>(v, red, 32, wid);
    __syncthreads();
    if (wid == 0) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = lane < nw ? red[q * 32 + lane] : make_float2(0.f, 0.f);
      warp_sum_store<NQ>(v, part + c.blk * 8, 1, 0);
    }
    if (!grid_sync(c)) return false;
    // one partial per lane of the first warps, then their sums
    const int ns = (c.nb + 31) >> 5;
    if (wid < ns) {
      const int i = lane + 32 * wid;
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = i < c.nb ? __ldcg(part + i * 8 + q) : make_float2(0.f, 0.f);
      warp_sum_store<NQ>(v, red, 32, wid);
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = lane < ns ? red[q * 32 + lane] : make_float2(0.f, 0.f);
      warp_sum_all<NQ>(v);
    }
    return true;
  }

  template <bool PK>
  static __device__ __forceinline__ void loop(const CoopArgs& ca) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ Scalars sc;
    __shared__ float2 red[5 * 32];
    __shared__ int bad;
    const PassArgs<float>& a = ca.one;
    const int tid = threadIdx.x;
    Ctx c;
    c.a = &a;
    c.cs = reinterpret_cast<CoopShared*>(ca.shared);
    c.work = reinterpret_cast<float2*>(smem_raw);
    c.R = ca.R;
    c.rows = ca.rows;
    c.nb = gridDim.x;
    c.blk = blockIdx.x;
    c.target = c.nb;  // the gathering's arrivals
    c.bad = &bad;
    c.magic = (65535 + c.R / 2) / (c.R / 2);
    float2* fld = c.work + Gm::work;  // [field][row slot][M/2] pairs: p, g, t, x (c or r)
    const int pl = c.R * (M / 2);
    float2 *fp = fld, *fg = fld + pl, *ft = fld + 2 * pl, *fx = fld + 3 * pl;
    for (int i = tid; i < (int)(sizeof(Scalars) / 4); i += Gm::NT)
      reinterpret_cast<int*>(&sc)[i] = __ldcg(reinterpret_cast<const int*>(a.sc) + i);
#ifdef BEM_DEBUG_CHECKS
    // Test hooks of debug builds: CTA 0 stays away from the gathering of the loop's
    // first launch (2) or second (3), or from the first grid barrier (1); the others'
    // waits run out (bounded).
    __syncthreads();
    const int away = blockIdx.x ? 0 : sc.inject == 1 ? 1 : sc.inject >= 2 && sc.coop_runs == sc.inject - 2 ? 2 : 0;
    if (away) {
      if (tid == 0) a.sc->inject = 0;
      if (away == 2) return;
    }
#endif
    if (tid == 0) {
      bad = 0;
      coop_arrive(c.cs, c.nb);
    }
    const int nx = a.pl.nx;
    const int b = tid / Gm::TR, t = tid % Gm::TR;
    const float us = (float)a.uscale;
    int par = 0;
    unsigned on = 0, S = 0;  // 8 bits per round of rows: on the grid, in the held set
    for (int r0 = 0, rd = 0; r0 < c.R; r0 += Gm::RPR, ++rd) {
      const int sl = r0 + b, row = c.blk * c.R + sl;
      if (!(b < Gm::RPR && sl < c.R)) continue;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (!FR::first_half(e)) continue;
        const int n = FR::n0(t, e);
        float vp[2] = {0, 0}, vg[2] = {0, 0}, vt[2] = {0, 0}, vx[2] = {0, 0};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = 2 * n + h;
          if (row < c.rows && col < nx) {
            const size_t j = (size_t)row * nx + col;
            const unsigned bit = 1u << (8 * rd + 2 * slot(e) + h);
            on |= bit;
            if (PK) {
              vp[h] = a.f.p[j];
              vx[h] = a.f.c[j];
              if (ca.resume) { vt[h] = a.f.t[j]; vg[h] = a.f.g[j]; }
            } else if (a.f.S[j]) {
              S |= bit;
              vp[h] = a.f.p[j];
              if (ca.resume) { vg[h] = a.f.g[j]; vt[h] = a.f.t[j]; vx[h] = a.f.r[j]; }
              else vx[h] = a.f.c[j];
            }
          }
        }
        const int i = sl * (M / 2) + n;
        if (n < M / 2) {
          fp[i] = make_float2(vp[0], vp[1]); fg[i] = make_float2(vg[0], vg[1]);
          ft[i] = make_float2(vt[0], vt[1]); fx[i] = make_float2(vx[0], vx[1]);
        }
      }
    }
    if (tid == 0 && !coop_all_came(c.cs)) bad = 1;
    __syncthreads();
    if (bad) return;  // not all CTAs are resident; nothing has been written
#ifdef BEM_DEBUG_CHECKS
    if (away) return;
#endif
    bool ok = true;
    // one transform per pass of this loop, whatever it is for (see resident.cuh)
    enum { kP, kT, kG };
    int step = PK ? kP : ca.resume ? kT : kG;
    for (int it = 0; it < ca.max_launch && !sc.done;) {
      const bool upd = sc.have_tau != 0;
      const float tau = (float)sc.tau, beta = (float)sc.beta;
      float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      float2 v5[5];
      phase_a(c, [&](int sl, int t_, float2* v) {
        const int rd = 8 * (sl / Gm::RPR);
        const unsigned onr = on >> rd, Sr = S >> rd;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          v[e] = make_float2(0.f, 0.f);
          if (!FR::first_half(e)) continue;
          const int i = sl * (M / 2) + FR::n0(t_, e);
          float2 pv = fp[i];
          if (step == kT) {
            float2 gv = fg[i], tv = ft[i];
            if (!PK && upd) {
              const float2 xv = fx[i];
              pv.x -= tau * tv.x; pv.y -= tau * tv.y;
              gv.x -= tau * xv.x; gv.y -= tau * xv.y;
              fp[i] = pv;
              fg[i] = gv;
            }
            const bool in0 = PK ? pv.x > 0.f : (Sr >> (2 * slot(e)) & 1) != 0;
            const bool in1 = PK ? pv.y > 0.f : (Sr >> (2 * slot(e) + 1) & 1) != 0;
            tv.x = in0 ? gv.x + beta * tv.x : 0.f;
            tv.y = in1 ? gv.y + beta * tv.y : 0.f;
            ft[i] = tv;
            v[e] = tv;
          } else {
            if (PK) {
              const float2 tv = ft[i], gv = fg[i];
              PIn<float> q;
              if (onr >> (2 * slot(e)) & 1) {
                q.p = pv.x; q.t = tv.x; q.g = gv.x;
                pv.x = pro_value<float, A_PK_P>(q, upd, tau, 0.f, acc);
              }
              if (onr >> (2 * slot(e) + 1) & 1) {
                q.p = pv.y; q.t = tv.y; q.g = gv.y;
                pv.y = pro_value<float, A_PK_P>(q, upd, tau, 0.f, acc);
              }
              if (upd) fp[i] = pv;
            }
            v[e] = pv;
          }
        }
      });
      if (!(ok = grid_sync(c))) break;
      phase_b(c);
      if (!(ok = grid_sync(c))) break;
      phase_c(c, [&](int sl, int t_, float2* v) {
        const int rd = 8 * (sl / Gm::RPR);
        const unsigned onr = on >> rd, Sr = S >> rd;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (!FR::first_half(e)) continue;
          const int i = sl * (M / 2) + FR::n0(t_, e);
          const float2 w = make_float2(us * v[e].x, us * v[e].y);
          if (PK) {
            const float2 pv = fp[i];
            if (step == kT) {
              const float2 gv = fg[i], tv = ft[i];
              if (pv.x > 0.f) { acc[0] += gv.x * tv.x; acc[1] += w.x * tv.x; }
              if (pv.y > 0.f) { acc[0] += gv.y * tv.y; acc[1] += w.y * tv.y; }
            } else {
              const float2 cv = fx[i];
              float2 gv = make_float2(0.f, 0.f);
              if (onr >> (2 * slot(e)) & 1) {
                gv.x = w.x + cv.x;
                if (pv.x > 0.f) { acc[3] += gv.x * gv.x; acc[4] += 1.f; }
              }
              if (onr >> (2 * slot(e) + 1) & 1) {
                gv.y = w.y + cv.y;
                if (pv.y > 0.f) { acc[3] += gv.y * gv.y; acc[4] += 1.f; }
              }
              fg[i] = gv;
            }
          } else {
            const bool in0 = Sr >> (2 * slot(e)) & 1, in1 = Sr >> (2 * slot(e) + 1) & 1;
            if (step == kT) {
              const float2 gv = fg[i], tv = ft[i];
              const float2 rv = make_float2(in0 ? w.x : 0.f, in1 ? w.y : 0.f);
              fx[i] = rv;
              acc[0] += rv.x * tv.x; acc[1] += rv.x * gv.x; acc[2] += rv.x * rv.x; acc[3] += gv.x * gv.x;
              acc[0] += rv.y * tv.y; acc[1] += rv.y * gv.y; acc[2] += rv.y * rv.y; acc[3] += gv.y * gv.y;
            } else {
              const float2 cv = fx[i];
              const float2 gv = make_float2(in0 ? w.x + cv.x : 0.f, in1 ? w.y + cv.y : 0.f);
              acc[0] += gv.x * gv.x + gv.y * gv.y;
              acc[1] += cv.x * cv.x + cv.y * cv.y;
              fg[i] = gv;
              fx[i] = make_float2(0.f, 0.f);
            }
          }
        }
      });
      if (!(ok = sum<PK ? 5 : 4>(c, acc, red, &par, v5))) break;
      if (tid < 32) {
        if (PK) {
          if (step == kP) finalize_pk_g(&sc, v5);
          else finalize_pk_r(&sc, v5);
        } else {
          if (step == kG) finalize_cg_g(&sc, v5);
          else finalize_cg_r(&sc, v5);
        }
      }
      __syncthreads();
      if (step == kT) ++it;
      step = PK && step == kT ? kP : kT;
    }
    if (!ok) {  // a wait ran out: give up together
      if (tid == 0 && a.kerr) atomicOr(a.kerr, 1u);
      return;
    }
    // a fixed-set solve may end with its last update pending
    const bool fin = !PK && sc.done && sc.have_tau;
    const float tau = (float)sc.tau;
    for (int r0 = 0; r0 < c.R; r0 += Gm::RPR) {
      const int sl = r0 + b, row = c.blk * c.R + sl;
      if (!(b < Gm::RPR && sl < c.R && row < c.rows)) continue;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (!FR::first_half(e)) continue;
        const int n = FR::n0(t, e), i = sl * (M / 2) + n;
        const float2 tv = ft[i], xv = fx[i];
        float2 pv = fp[i], gv = fg[i];
        if (fin) {
          pv.x -= tau * tv.x; pv.y -= tau * tv.y;
          gv.x -= tau * xv.x; gv.y -= tau * xv.y;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = 2 * n + h;
          if (col >= nx) continue;
          const size_t j = (size_t)row * nx + col;
          a.f.p[j] = h ? pv.y : pv.x;
          a.f.g[j] = h ? gv.y : gv.x;
          a.f.t[j] = h ? tv.y : tv.x;
          if (!PK) a.f.r[j] = h ? xv.y : xv.x;
        }
      }
    }
    // rows past c.rows hold no pressure (nor, in a loop that goes on, anything else)
    for (size_t i = (size_t)c.rows * nx + (size_t)blockIdx.x * Gm::NT + tid; i < (size_t)a.pl.ny * nx;
         i += (size_t)c.nb * Gm::NT) {
      a.f.p[i] = 0.f;
      if (!sc.done) a.f.g[i] = a.f.t[i] = a.f.r[i] = 0.f;
    }
    if (blockIdx.x == 0) {  // the scalars, all but the sticky error word
      __syncthreads();
      if (tid == 0) {
        sc.coop_runs += 1;
        if (fin) sc.have_tau = 0;
      }
      __syncthreads();
      for (int i = tid; i < (int)(offsetof(Scalars, kerr) / 4); i += Gm::NT)
        reinterpret_cast<int*>(a.sc)[i] = reinterpret_cast<const int*>(&sc)[i];
    }
  }
};

template <int LM, int LP, bool PK>
__global__ void __launch_bounds__(CoopGeo<LM, LP>::NT, 1) k_coop(const __grid_constant__ CoopArgs r) {
  Coop<LM, LP>::template loop<PK>(r);
}

#define BEM_COOP_CASES(X) X(8, 9) X(8, 10) X(8, 11) X(9, 9) X(9, 10) X(9, 11) X(10, 9) X(10, 10) X(10, 11)

template <int LM, int LP>
constexpr size_t coop_smem(int R) { return 8 * (size_t)CoopGeo<LM, LP>::work + 16 * (size_t)R * CoopGeo<LM, LP>::M; }

// CTAs and rows per CTA of the loop over `rows` rows: as many CTAs as give every
// one a round of columns, at most one per SM; an even number of rows each, so
// that W is read and written in 16-byte pairs.  False where a CTA's share of the
// rows does not fit its registers' bit masks or its shared memory (a device or
// partition of few SMs: 1024 rows of 1024 points need 128).
constexpr size_t kCoopSmemMax = 224 * 1024;  // an SM's 227 KB less the static part
template <int LM, int LP>
inline bool coop_shape(int rows, int nsm, int* nb, int* R) {
  using Gm = CoopGeo<LM, LP>;
  *nb = std::min(std::min(nsm, kCoopMaxCtas), (Gm::M + 1 + Gm::CPR - 1) / Gm::CPR);
  if (*nb < 1) return false;
  *R = 2 * std::max(1, (rows + 2 * *nb - 1) / (2 * *nb));
  return *R <= Gm::RMAX && coop_smem<LM, LP>(*R) <= kCoopSmemMax;
}

template <bool PK>
cudaError_t launch_coop_kind(CoopArgs r, int lm, int lp, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // a fresh barrier and gathering for every launch
  cudaError_t e = cudaMemsetAsync(r.shared, 0, offsetof(CoopShared, pad), s);
  if (e != cudaSuccess) return e;
  switch (lm * 16 + lp) {
#define BEM_CASE(LM, LP)                                                     \
  case LM * 16 + LP: {                                                       \
    int nb = 0;                                                              \
    if (!coop_shape<LM, LP>(r.rows, r.one.pl.nsm, &nb, &r.R)) return cudaErrorInvalidValue; \
    cfg.gridDim = dim3(nb);                                                  \
    cfg.blockDim = dim3(CoopGeo<LM, LP>::NT);                                \
    cfg.dynamicSmemBytes = coop_smem<LM, LP>(r.R);                           \
    return cudaLaunchKernelEx(&cfg, k_coop<LM, LP, PK>, r);                  \
  }
    BEM_COOP_CASES(BEM_CASE)
#undef BEM_CASE
  }
  return cudaErrorInvalidValue;
}

template <bool PK>
cudaError_t coop_setup_kind() {
  cudaError_t e = cudaSuccess, r;
#define BEM_CASE(LM, LP) \
  if ((r = set_smem_max(k_coop<LM, LP, PK>, 227 * 1024)) != cudaSuccess && e == cudaSuccess) e = r;
  BEM_COOP_CASES(BEM_CASE)
#undef BEM_CASE
  return e;
}

}  // namespace bem
