// CG loops of small grids inside one thread-block cluster (FP32 path).
//
// On a grid of at most 256 x 256 elements one pass of the transform is a few
// microseconds of latency -- launch, scalar reads, staging, the last CTA's sums
// -- around well under a microsecond of work, three (fixed-set CG) or six
// (Polonsky-Keer) times per iteration.  Here a whole solve's loop is one launch
// of one cluster of CS CTAs that keeps everything on chip:
//   - CTA r owns the grid rows r R .. r R + R - 1; a thread keeps its eight
//     elements of p, g, t and r (or c) in registers for the whole loop;
//   - it also owns the columns kx = r Q .. r Q + Q - 1 of the half spectrum;
//   - the two transposes of a transform are stores into the owners' shared
//     memory (distributed shared memory), each followed by a cluster barrier:
//     rows' spectra go to the column owners, column results to the row owners;
//   - sums are formed per CTA as float-float pairs, sent to every CTA of the
//     cluster, and added there in the same order, so that every CTA takes the
//     same decision from its own copy of the solve's scalars.
// The arithmetic is that of the passes (FftC stages, the same prologues and
// epilogues); only the order of the partial sums differs.
//
// Bound by latency: about 12 barriers and 10 FFT stages per transform.  Measured
// (GB300, per Polonsky-Keer iteration, two transforms): 32 x 32 10 us, 128 x 128
// 15, 256 x 256 30, as passes 29, 34 and 36; a fixed-set iteration takes half.
#pragma once
#include "conv_kernels.cuh"

namespace bem {

constexpr int res_lg(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l > 6 ? 6 : l;
}

// Geometry of the loop for row transforms of length M = 2^LM (grids up to M
// columns) and column transforms of length 2^LP (grids up to 2^LP / 2 rows).
// Sixteen CTAs, the largest cluster, unless the grid has fewer rows than fill
// them; column rounds so that a CTA has at most 576 threads (112 registers).
template <int LM, int LP>
struct ResGeo {
  static constexpr int M = 1 << LM, P = 1 << LP, NY = P / 2;
  static constexpr int CS = LM >= 6 || LP >= 7 ? 16 : 8;
  static constexpr int R = NY / CS >= 2 ? NY / CS : 2;        // rows per CTA (even)
  static constexpr int Q = (M + CS) / CS;                     // columns per CTA
  static constexpr int TR = M / 8, TC = P / 8;                // threads per row / column
  static constexpr int NR = (Q * TC + 575) / 576;             // column rounds
  static constexpr int CR = (Q + NR - 1) / NR;                // columns per round
  static constexpr int NT0 = R * TR > CR * TC ? R * TR : CR * TC;
  static constexpr int NT = NT0 < 64 ? 64 : (NT0 + 31) / 32 * 32;
  static constexpr int LR = res_lg(R);
  static constexpr int RS = M + kGeo8[LM - 3].pad[res_lg(R)];     // row pitch (complex)
  static constexpr int CZ = P + kGeo8[LP - 3].pad[res_lg(CR)];    // column pitch
  static constexpr int CP = NY + (R < 16 ? R : 16);           // pitch of a received column
  // float2 offsets
  static constexpr int o_rowz = 0;
  static constexpr int o_rowin = (o_rowz + R * RS + 1) & ~1;
  static constexpr int o_colin = (o_rowin + (M + 1) * R + 1) & ~1;
  static constexpr int o_colz = (o_colin + Q * CP + 1) & ~1;
  static constexpr size_t smem = 8 * (size_t)(o_colz + CR * CZ);
};

__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cl_map(const void* p, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_st2(unsigned addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cl_st4(unsigned addr, float2 v, float2 w) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(w.x),
               "f"(w.y)
               : "memory");
}

__device__ __forceinline__ float2 ff_xor(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// Sums of NQ (2, 4 or 5) float-float values over the lanes of a warp.  The first
// levels scatter: a lane passes on half of its values and keeps the other half,
// so that two or four sums take six additions a lane instead of ten or twenty (a
// float-float addition is ten instructions, and every warp of the CTA forms
// these sums).  The lane's own quantity, warp_sum_q(lane), is
// returned in v[0], a fifth one in v[4] of every lane; the additions commute, so
// all lanes of a quantity hold the same bits.
template <int NQ>
__device__ __forceinline__ int warp_sum_q(int lane) { return NQ == 2 ? lane >> 4 : lane >> 3; }
template <int NQ>
__device__ __forceinline__ void warp_sum_mine(float2* v) {
  const int lane = threadIdx.x & 31;
  const bool h4 = lane & 16, h3 = lane & 8;
  if (NQ == 5) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[NQ - 1] = ff_add(v[NQ - 1], ff_xor(v[NQ - 1], o));
  }
  float2 a;
  if constexpr (NQ == 2) {
    a = ff_add(h4 ? v[1] : v[0], ff_xor(h4 ? v[0] : v[1], 16));
    a = ff_add(a, ff_xor(a, 8));
  } else {
    const float2 x = ff_add(h4 ? v[2] : v[0], ff_xor(h4 ? v[0] : v[2], 16));
    const float2 y = ff_add(h4 ? v[3] : v[1], ff_xor(h4 ? v[1] : v[3], 16));
    a = ff_add(h3 ? y : x, ff_xor(h3 ? x : y, 8));
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) a = ff_add(a, ff_xor(a, o));
  v[0] = a;
}
// ... the totals in every lane
template <int NQ>
__device__ __forceinline__ void warp_sum_all(float2* v) {
  warp_sum_mine<NQ>(v);
  const float2 a = v[0];
  constexpr int W = NQ == 2 ? 16 : 8, N = NQ == 2 ? 2 : 4;
#pragma unroll
  for (int q = 0; q < N; ++q) v[q] = make_float2(__shfl_sync(0xffffffffu, a.x, q * W), __shfl_sync(0xffffffffu, a.y, q * W));
}
// ... one warp's sums into red[q * stride + i] (leading lanes write)
template <int NQ>
__device__ __forceinline__ void warp_sum_store(float2* v, float2* red, int stride, int i) {
  warp_sum_mine<NQ>(v);
  const int lane = threadIdx.x & 31;
  constexpr int W = NQ == 2 ? 16 : 8;
  if ((lane & (W - 1)) == 0) red[warp_sum_q<NQ>(lane) * stride + i] = v[0];
  if (NQ == 5 && lane == 1) red[4 * stride + i] = v[NQ - 1];
}

// The scalar decisions of pass_c_finalize taken by one warp on sums that every
// lane holds.  FP64 instructions are slow one after another and occupy the pipe
// by active lanes (a whole warp's division: over 2 us), so conversions and
// divisions run side by side in as few lanes as there are values.
__device__ __forceinline__ bool fin64(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ void finalize_cg_r(Scalars* sc, const float2* v) {
  const int lane = threadIdx.x & 31;
  double d = 0.0, rd = 0.0;
  if (lane < 4) {
    d = ff_to_double(lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : v[3]);
    if (lane == 0 || lane == 3) rd = 1.0 / d;
  }
  __syncwarp();
  const double str = __shfl_sync(0xffffffffu, d, 0), sgr = __shfl_sync(0xffffffffu, d, 1);
  const double srr = __shfl_sync(0xffffffffu, d, 2), G = __shfl_sync(0xffffffffu, d, 3);
  const double rstr = __shfl_sync(0xffffffffu, rd, 0), rG = __shfl_sync(0xffffffffu, rd, 3);
  if (lane) return;
  const double stop2 = sc->stop2;
  const int iter = sc->iter, loops = sc->loops + 1;
  int done = 0, status = SC_OK, have = 0;
  double tau = 0.0, beta = 0.0, gn = G;
  if (!fin64(str) || !fin64(G) || !fin64(sgr) || !fin64(srr)) {
    status = SC_NUMERIC;
    done = 1;
  } else if (G <= stop2 || str <= 0.0) {
    done = 1;
  } else if (iter >= sc->max_iter) {
    status = SC_NOCONV;
    done = 1;
  } else {
    tau = G * rstr;
    gn = fma(tau, fma(tau, srr, -2.0 * sgr), G);
    if (gn < 0.0) gn = 0.0;
    beta = gn * rG;
    have = 1;
    if (gn <= stop2) done = 1;  // converged once this update is applied
  }
  if (!done && loops >= sc->max_loops) {
    status = SC_NOCONV;
    done = 1;
  }
  sc->loops = loops;
  sc->str = str;
  sc->G = gn;
  sc->have_tau = have;
  if (have) {
    sc->tau = tau;
    sc->beta = beta;
    sc->iter = iter + 1;
  }
  if (status != SC_OK) sc->status = status;
  if (done) sc->done = 1;
}
// v: |g|^2, |c|^2 on the set
__device__ __forceinline__ void finalize_cg_g(Scalars* sc, const float2* v) {
  if (threadIdx.x & 31) return;
  const double s2[4] = {ff_to_double(v[0]), ff_to_double(v[1]), 0, 0}, s3[3] = {0, 0, 0};
  pass_c_finalize<float, C_CG_G>(sc, s2, s3, CgPre{});
}
// v: sum |dp|, sum p, #overlap, sum g^2, #(p > 0)
__device__ __forceinline__ void finalize_pk_g(Scalars* sc, const float2* v) {
  const int lane = threadIdx.x & 31;
  double d = 0.0, q = 0.0;
  if (lane < 5) d = ff_to_double(lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : lane == 3 ? v[3] : v[4]);
  __syncwarp();
  const double sp = __shfl_sync(0xffffffffu, d, 1), G = __shfl_sync(0xffffffffu, d, 3);
  if (lane < 2) q = (lane == 0 ? d : G) / (lane == 0 ? sp : sc->G_old);  // eps, G / G_old
  __syncwarp();
  const double nol = __shfl_sync(0xffffffffu, d, 2), nic = __shfl_sync(0xffffffffu, d, 4);
  const double ratio = __shfl_sync(0xffffffffu, q, 1);
  if (lane) return;
  int done = 0;
  if (sc->have_tau) {
    sc->sum_dp = d;
    sc->sum_p = sp;
    sc->n_ol = nol;
    const int iter = sc->iter += 1;
    const double eps = sp > 0.0 ? q : 0.0;
    sc->eps = eps;
    sc->delta = nol > 0.0 ? 0.0 : 1.0;
    if (!fin64(eps) || !fin64(G)) { sc->status = SC_NUMERIC; done = 1; }
    else if (eps < sc->tol) done = 1;
    else if (iter >= sc->max_iter) { sc->status = SC_NOCONV; done = 1; }
    if (!done) {
      if (iter == 1 || eps < 0.5 * sc->eps_min) { sc->eps_min = eps; sc->it_min = iter; }
      else if (iter - sc->it_min > kStall) { sc->status = SC_STALL; done = 1; }
    }
  }
  sc->n_ic = nic;
  sc->G = G;
  if (!done) {
    if (nic == 0.0 || G == 0.0) done = 1;
    else { sc->beta = sc->delta > 0.0 ? ratio : 0.0; sc->G_old = G; }
  }
  if (done) sc->done = 1;
}
// v: sum g t, sum r t over p > 0
__device__ __forceinline__ void finalize_pk_r(Scalars* sc, const float2* v) {
  const int lane = threadIdx.x & 31;
  double d = 0.0;
  if (lane < 2) d = ff_to_double(lane == 0 ? v[0] : v[1]);
  __syncwarp();
  const double sgt = __shfl_sync(0xffffffffu, d, 0), srt = __shfl_sync(0xffffffffu, d, 1);
  if (lane) return;
  const double s2[4] = {sgt, srt, 0, 0}, s3[3] = {0, 0, 0};
  pass_c_finalize<float, C_PK_R>(sc, s2, s3, CgPre{});
}

template <int LM, int LP>
struct Resident {
  using Gm = ResGeo<LM, LP>;
  using FR = FftC<float, LM>;
  using FC = FftC<float, LP>;
  static constexpr int M = Gm::M, P = Gm::P, R = Gm::R, Q = Gm::Q, CS = Gm::CS;

  // register slot pair (0..3) of stage-0 element e (first half only)
  static __device__ __forceinline__ constexpr int slot(int e) {
    return FR::R0 == 0 ? e : FR::R0 == 2 ? (e >> 2) * 2 + (e & 1) : e >> 1;
  }
  static __device__ __forceinline__ void col_sync(int c) {
    if (Gm::TC <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(c + 1), "r"(Gm::TC) : "memory");
  }

  // u = K*x scaled by us, x and u in the threads' register slots (zero off the grid).
  static __device__ __forceinline__ void conv(const PassArgs<float>& a, float2* sm, unsigned rank, int ny,
                                              const float* x, float* u, float us) {
    const int tid = threadIdx.x;
    const int b = tid / Gm::TR, t = tid % Gm::TR;
    const bool ra = b < R;
    float2* rowz = sm + Gm::o_rowz;
    float2* rowin = sm + Gm::o_rowin;
    float2* colin = sm + Gm::o_colin;
    const float2* twA = reinterpret_cast<const float2*>(a.twA);
    const float2* twB = reinterpret_cast<const float2*>(a.twB);
    const float2* tws = reinterpret_cast<const float2*>(a.twS);
    const int* sp = a.spA;
    float2* buf = rowz + (ra ? b : 0) * Gm::RS;
    float2 v[8];
    // rows: forward (a row's threads are lanes of one warp)
    if (ra) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        v[e] = FR::first_half(e) ? make_float2(x[2 * slot(e)], x[2 * slot(e) + 1]) : make_float2(0.f, 0.f);
      FR::stage0_fwd(v, t, twA);
#pragma unroll
      for (int e = 0; e < 8; ++e) buf[FR::ix0(t, e)] = v[e];
    }
    __syncwarp();
#pragma unroll
    for (int ls = FR::LS_TOP; ls >= 0; ls -= 3) {
      if (ra) FR::dif(buf, t, ls, twA);
      __syncwarp();
    }
    __syncthreads();
    // split into half spectra, two rows per item, to the columns' owners
    {
      constexpr int LR = Gm::LR - 1;
      const int y0 = (int)rank * R;
      const int items = y0 < Gm::NY ? (M / 2 + 1) << LR : 0;  // a cluster larger than the rows: idle ranks
      for (int idx = tid; idx < items; idx += Gm::NT) {
        const int k = idx >> LR, bb = 2 * (idx & ((1 << LR) - 1));
        const float2* s0 = rowz + bb * Gm::RS;
        const float2* s1 = s0 + Gm::RS;
        float2 xk0, xm0, xk1, xm1;
        if (k == 0) {
          const float2 z0 = s0[0], z1 = s1[0];
          xk0 = make_float2(z0.x + z0.y, 0.f);
          xm0 = make_float2(z0.x - z0.y, 0.f);
          xk1 = make_float2(z1.x + z1.y, 0.f);
          xm1 = make_float2(z1.x - z1.y, 0.f);
        } else {
          const int pk = __ldg(sp + k), pm = __ldg(sp + M - k);
          const float2 w = __ldg(tws + k);
          split_two<float>(s0, pk, pm, w, xk0, xm0);
          split_two<float>(s1, pk, pm, w, xk1, xm1);
        }
        const int km = k == 0 ? M : M - k;
        if (!bem_check(k / Q < CS && km / Q < CS && y0 + bb + 1 < Gm::CP, a.kerr)) continue;
        cl_st4(cl_map(colin + (k % Q) * Gm::CP + y0 + bb, k / Q), xk0, xk1);
        if (km != k) cl_st4(cl_map(colin + (km % Q) * Gm::CP + y0 + bb, km / Q), xm0, xm1);
      }
    }
    cl_sync();
    // columns: forward, spectrum multiply, inverse
    {
      constexpr int L = P, L8 = Gm::TC, hyq = L / 2 + 1;
      const int c = tid / Gm::TC, tc = tid % Gm::TC;
      const int* spB = a.spB;
      float2* cz = sm + Gm::o_colz + (c < Gm::CR ? c : 0) * Gm::CZ;
#pragma unroll 1
      for (int rd = 0; rd < Gm::NR; ++rd) {
        const int cl = rd * Gm::CR + c, kx = (int)rank * Q + cl;
        const bool ca = c < Gm::CR && cl < Q && kx <= M;
        if (Gm::TC > 32 && !ca) continue;  // whole column groups: the others' barriers are their own
        const float2* in = colin + (ca ? cl : 0) * Gm::CP;
        if (ca) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            v[e] = make_float2(0.f, 0.f);
            if (!FC::first_half(e)) continue;
            const int y = FC::n0(tc, e);
            if (y < ny) v[e] = in[y];
          }
          FC::stage0_fwd(v, tc, twB);
#pragma unroll
          for (int e = 0; e < 8; ++e) cz[FC::ix0(tc, e)] = v[e];
        }
        col_sync(c);
#pragma unroll
        for (int ls = FC::LS_TOP; ls >= 3; ls -= 3) {
          if (ca) FC::dif(cz, tc, ls, twB);
          col_sync(c);
        }
        if (ca) {
          const int sp0 = __ldg(spB + tc);
          const float* kc = a.khat + (size_t)kx * hyq;
          float kf[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int ky = tc + q * L8;
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
        col_sync(c);
#pragma unroll
        for (int ls = 3; ls <= FC::LS_TOP; ls += 3) {
          if (ca) FC::dit(cz, tc, ls, twB);
          col_sync(c);
        }
        if (ca) {
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = cz[FC::ix0(tc, e)];
          FC::stage0_inv(v, tc, twB);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            if (!FC::first_half(e)) continue;
            const int y = FC::n0(tc, e);
            if (y < ny && bem_check(kx <= M && y / R < CS, a.kerr)) cl_st2(cl_map(rowin + kx * R + y % R, y / R), v[e]);
          }
        }
      }
    }
    cl_sync();
    // rows: rebuild the packed spectra, inverse
    {
      constexpr int LR = Gm::LR;
      for (int idx = tid; idx < (M / 2 + 1) << LR; idx += Gm::NT) {
        const int k = idx >> LR, bb = idx & (R - 1);
        const float2 xk = rowin[(k << LR) + bb], xm = rowin[((M - k) << LR) + bb];
        float2* s = rowz + bb * Gm::RS;
        const float2 wk = conj<float>(__ldg(tws + k));
        const float2 E = add<float>(xk, conj<float>(xm));
        const float2 O = mul<float>(sub<float>(xk, conj<float>(xm)), wk);
        s[__ldg(sp + k)] = add<float>(E, mul_si<float, 1>(O));
        if (k != 0 && k != M - k) {
          const float2 wm = make_float2(-wk.x, wk.y);
          const float2 E2 = add<float>(xm, conj<float>(xk));
          const float2 O2 = mul<float>(sub<float>(xm, conj<float>(xk)), wm);
          s[__ldg(sp + M - k)] = add<float>(E2, mul_si<float, 1>(O2));
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int ls = 0; ls <= FR::LS_TOP; ls += 3) {
      if (ra) FR::dit(buf, t, ls, twA);
      __syncwarp();
    }
    if (ra) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = buf[FR::ix0(t, e)];
      FR::stage0_inv(v, t, twA);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (!FR::first_half(e)) continue;
        u[2 * slot(e)] = us * v[e].x;
        u[2 * slot(e) + 1] = us * v[e].y;
      }
    }
  }

  // Sums over the cluster of NQ per-thread values, the same in every CTA: in all
  // lanes of warp 0.  slots: CS x 8 float2 in shared memory, red: NQ per warp.
  template <int NQ>
  static __device__ __forceinline__ void sum(const float* acc, float2* red, float2* slots, unsigned rank, float2* v) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int nw = Gm::NT / 32;
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = make_float2(acc[q], 0.f);
    warp_sum_store<NQ>(v, red, nw, wid);
    __syncthreads();
    if (wid == 0) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = lane < nw ? red[q * nw + lane] : make_float2(0.f, 0.f);
      warp_sum_all<NQ>(v);
      if (lane < CS) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) cl_st2(cl_map(slots + rank * 8 + q, lane), v[q]);
      }
    }
    cl_sync();
    if (wid == 0) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = lane < CS ? slots[lane * 8 + q] : make_float2(0.f, 0.f);
      warp_sum_all<NQ>(v);
    }
  }

  template <bool PK>
  static __device__ __forceinline__ void loop(const ResArgs& ra_) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ Scalars sc;
    __shared__ float2 red[5 * (Gm::NT / 32)];
    __shared__ float2 slots[CS * 8];
    float2* sm = reinterpret_cast<float2*>(smem_raw);
    const PassArgs<float>& a = ra_.arr ? ra_.arr[blockIdx.y] : ra_.one;
    const unsigned rank = cl_rank();
    const int tid = threadIdx.x;
    for (int i = tid; i < (int)(sizeof(Scalars) / 4); i += Gm::NT)
      reinterpret_cast<int*>(&sc)[i] = reinterpret_cast<const volatile int*>(a.sc)[i];
    const int nx = a.pl.nx, ny = a.pl.ny;
    const int b = tid / Gm::TR, t = tid % Gm::TR;
    const int row = (int)rank * R + b;
    const bool act = b < R && row < ny;
    const float us = (float)a.uscale;
    // rows past the grid and columns past the half spectrum are never written: zero
    for (int i = tid; i < Gm::o_colz; i += Gm::NT) sm[i] = make_float2(0.f, 0.f);
    __syncthreads();
#ifdef BEM_DEBUG_CHECKS
    // Test hook of debug builds: a wait that nothing completes runs out (bounded).
    if (sc.inject == 1) {
      __shared__ unsigned long long never;
      cl_sync();
      if (rank == 0 && tid == 0) {
        a.sc->inject = 0;
        mbar_init(&never, 1);
        if (!mbar_wait(&never, 0) && a.kerr) atomicOr(a.kerr, 1u);
      }
      return;
    }
#endif
    float p[8], g[8], tt[8], x[8];  // x: c (Polonsky-Keer) or r
    unsigned S = 0, on = 0;         // held elements; elements of the grid
    float u[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!FR::first_half(e)) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = 2 * slot(e) + h, col = 2 * FR::n0(t, e) + h;
        p[i] = g[i] = tt[i] = x[i] = u[i] = 0.f;
        if (act && col < nx) {
          const size_t j = (size_t)row * nx + col;
          on |= 1u << i;
          if (PK) {
            p[i] = a.f.p[j];
            x[i] = a.f.c[j];
            if (ra_.resume) { tt[i] = a.f.t[j]; g[i] = a.f.g[j]; }
          } else if (a.f.S[j]) {
            S |= 1u << i;
            p[i] = a.f.p[j];
            if (ra_.resume) { g[i] = a.f.g[j]; tt[i] = a.f.t[j]; x[i] = a.f.r[j]; }
            else x[i] = a.f.c[j];
          }
        }
      }
    }
    cl_sync();  // every CTA's buffers are cleared before anyone stores into them
    // One transform per pass of this loop, whatever it is for, so that its code
    // exists once (the loop's instructions are fetched for a few warps only).
    //   PK: kP updates p and forms the gap, kT the direction and its transform;
    //   CG: kG forms the initial residual, kT is an iteration.
    enum { kP, kT, kG };
    int step = PK ? kP : ra_.resume ? kT : kG;
    for (int it = 0; it < ra_.max_launch && !sc.done;) {
      const bool upd = sc.have_tau != 0;
      const float tau = (float)sc.tau, beta = (float)sc.beta;
      float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, y[8];
      float2 v5[5];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (step == kT) {
          if (!PK && upd) { p[i] -= tau * tt[i]; g[i] -= tau * x[i]; }
          tt[i] = (PK ? p[i] > 0.f : (S >> i & 1) != 0) ? g[i] + beta * tt[i] : 0.f;
          y[i] = tt[i];
        } else {
          if (PK && (on >> i & 1)) {
            PIn<float> q;
            q.p = p[i]; q.t = tt[i]; q.g = g[i];
            p[i] = pro_value<float, A_PK_P>(q, upd, tau, 0.f, acc);
          }
          y[i] = p[i];
        }
      }
      conv(a, sm, rank, ny, y, u, us);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (PK) {
          if (step == kT) {
            if (p[i] > 0.f) { acc[0] += g[i] * tt[i]; acc[1] += u[i] * tt[i]; }
          } else if (on >> i & 1) {
            g[i] = u[i] + x[i];
            if (p[i] > 0.f) { acc[3] += g[i] * g[i]; acc[4] += 1.f; }
          }
        } else if (step == kT) {
          x[i] = S >> i & 1 ? u[i] : 0.f;
          acc[0] += x[i] * tt[i];
          acc[1] += x[i] * g[i];
          acc[2] += x[i] * x[i];
          acc[3] += g[i] * g[i];
        } else {
          g[i] = S >> i & 1 ? u[i] + x[i] : 0.f;
          acc[0] += g[i] * g[i];
          acc[1] += x[i] * x[i];
          x[i] = 0.f;
        }
      }
      sum<PK ? 5 : 4>(acc, red, slots, rank, v5);
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
    // a fixed-set solve may end with its last update pending
    const bool fin = !PK && sc.done && sc.have_tau;
    const float tau = (float)sc.tau;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!FR::first_half(e)) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = 2 * slot(e) + h, col = 2 * FR::n0(t, e) + h;
        if (!(on >> i & 1)) continue;
        const size_t j = (size_t)row * nx + col;
        a.f.p[j] = fin ? p[i] - tau * tt[i] : p[i];
        a.f.g[j] = fin ? g[i] - tau * x[i] : g[i];
        a.f.t[j] = tt[i];
        if (!PK) a.f.r[j] = x[i];
      }
    }
    __syncthreads();
    if (tid == 0 && fin) sc.have_tau = 0;
    __syncthreads();
    // CTA 0 returns the scalars (all but the sticky error word)
    if (rank == 0)
      for (int i = tid; i < (int)(offsetof(Scalars, kerr) / 4); i += Gm::NT)
        reinterpret_cast<int*>(a.sc)[i] = reinterpret_cast<const int*>(&sc)[i];
    cl_sync();  // no CTA leaves while another may still store into it
  }
};

template <int LM, int LP, bool PK>
__global__ void __launch_bounds__(ResGeo<LM, LP>::NT, 1) k_resident(const __grid_constant__ ResArgs r) {
  Resident<LM, LP>::template loop<PK>(r);
}

#define BEM_RES_CASES(X) \
  X(4, 5) X(4, 6) X(4, 7) X(4, 8) X(4, 9) X(5, 5) X(5, 6) X(5, 7) X(5, 8) X(5, 9) X(6, 5) X(6, 6) X(6, 7) X(6, 8) \
  X(6, 9) X(7, 5) X(7, 6) X(7, 7) X(7, 8) X(7, 9) X(8, 5) X(8, 6) X(8, 7) X(8, 8) X(8, 9)

template <bool PK>
cudaError_t launch_resident_kind(const ResArgs& r, int lm, int lp, int n, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  switch (lm * 16 + lp) {
#define BEM_CASE(LM, LP)                                                     \
  case LM * 16 + LP: {                                                       \
    using Gm = ResGeo<LM, LP>;                                               \
    at[0].val.clusterDim.x = Gm::CS;                                         \
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;                     \
    cfg.gridDim = dim3(Gm::CS, n);                                           \
    cfg.blockDim = dim3(Gm::NT);                                             \
    cfg.dynamicSmemBytes = Gm::smem;                                         \
    return cudaLaunchKernelEx(&cfg, k_resident<LM, LP, PK>, r);              \
  }
    BEM_RES_CASES(BEM_CASE)
#undef BEM_CASE
  }
  return cudaErrorInvalidValue;
}

// Whether a sixteen-CTA cluster of the largest kernel can run on this device.
template <bool PK>
bool resident_runs_kind() {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(ResGeo<8, 9>::NT);
  cfg.dynamicSmemBytes = ResGeo<8, 9>::smem;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_resident<8, 9, PK>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n > 0;
}

// Opt the kernels into their shared memory and sixteen-CTA clusters.
template <bool PK>
cudaError_t resident_setup_kind() {
  cudaError_t e = cudaSuccess, r;
#define BEM_CASE(LM, LP)                                                                                        \
  if ((r = cudaFuncSetAttribute(k_resident<LM, LP, PK>, cudaFuncAttributeMaxDynamicSharedMemorySize,            \
                                (int)ResGeo<LM, LP>::smem)) != cudaSuccess && e == cudaSuccess) e = r;          \
  if ((r = cudaFuncSetAttribute(k_resident<LM, LP, PK>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) !=  \
          cudaSuccess && e == cudaSuccess) e = r;
  BEM_RES_CASES(BEM_CASE)
#undef BEM_CASE
  return e;
}

}  // namespace bem
