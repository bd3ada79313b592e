// fr_stage_fx.cuh -- element and trace kernels of the FP64 form (arXiv 2306.06744, Sec. 2.1), with
// their contractions in block fixed point (fr_fixed.cuh).
#pragma once

#include "fr_fixed.cuh"
#include "fr_kernels.cuh"

namespace frg {

// Operator tables of the fixed-point contractions (passed by value: constant bank, copied to shared
// memory by the kernels because threads of a warp read different rows)
struct TraceFx {
  int2 lm[NPMAX], lp[NPMAX];
  int kt;  // scale of the entries
};
struct OpsFx {
  int2 Dt[NPMAX][NPMAX], gLh[NPMAX], gRh[NPMAX];
  int kd;                    // scale of the derivative and its correction
  TraceFx tr;
  double D[NPMAX][NPMAX];    // plain derivative (density-gradient indicator, FP64)
  double gm1, ngmh;          // gamma - 1, -(gamma - 1)/2
};
inline TraceFx make_trace_fx(int p, const DevOps& o) {
  TraceFx r{};
  double st[2] = {0.0, 0.0};
  for (int i = 0; i <= p; ++i) {
    st[0] += fabs(o.lm[i]);
    st[1] += fabs(o.lp[i]);
  }
  r.kt = fx_scale(st[0] > st[1] ? st[0] : st[1]);
  for (int i = 0; i <= p; ++i) {
    r.lm[i] = fx_coef(o.lm[i], r.kt);
    r.lp[i] = fx_coef(o.lp[i], r.kt);
  }
  return r;
}
// gLh, gRh carry the factor 1/2 of the doubled common flux
inline OpsFx make_ops_fx(int dim, int p, const DevOps& o, double gamma) {
  OpsFx r{};
  const int n = p + 1;
  double sd = 0.0;
  for (int i = 0; i < n; ++i) {
    double s = 0.5 * (fabs(o.gL[i]) + fabs(o.gR[i]));
    for (int j = 0; j < n; ++j) s += fabs(o.Dt[i][j]);
    sd = s > sd ? s : sd;
  }
  r.kd = fx_scale(dim * sd);  // one accumulator sums the terms of all axes
  r.tr = make_trace_fx(p, o);
  for (int i = 0; i < n; ++i) {
    r.gLh[i] = fx_coef(0.5 * o.gL[i], r.kd);
    r.gRh[i] = fx_coef(0.5 * o.gR[i], r.kd);
    for (int j = 0; j < n; ++j) {
      r.Dt[i][j] = fx_coef(o.Dt[i][j], r.kd);
      r.D[i][j] = o.D[i][j];
    }
  }
  r.gm1 = gamma - 1.0;
  r.ngmh = -0.5 * (gamma - 1.0);
  return r;
}

// Place of point i in an element's staged state.  At 3D p = 3 the lines along x of 16 lanes start 32
// bytes apart, four to a bank, and so do those along y in different planes: x and y are exclusive-ored
// with the plane's index, which spreads both over all banks.
template <int DIM, int NP>
__device__ __forceinline__ constexpr int fx_place(int i) {
  return DIM == 3 && NP == 4 ? i ^ ((i >> 4) * 5) : i;
}

// Traces of the block's elements from their fixed-point state sv[le][v][place of i] with group exponents
// se[le][group]: one thread per (element, face, face point), all variables.  need (nullable): only
// elements with a non-zero entry.
template <int DIM, int NP>
__device__ __forceinline__ void fx_traces(const int2* sv, const uint32_t* se, const int2* slm, const int2* slp, int kt,
                                          int ne, const int8_t* need, double* to) {
  using S = Sz<DIM, NP>;
  constexpr int N = S::N, NV = S::NV, NF = S::NF, EU = S::EU, EF = S::EF, FQ = S::NFC * NF;
  for (int k = threadIdx.x; k < ne * FQ; k += blockDim.x) {
    const int le = k / FQ, r = k % FQ;
    if (need && !need[le]) continue;
    const int f = r / NF, q = r % NF;
    const int2* lf = (f & 1) ? slp : slm;
    int2 c[NP];
    int pts[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      c[j] = lf[j];
      pts[j] = le * EU + fx_place<DIM, NP>(line_pt<DIM, NP>(f >> 1, q, j));
    }
    double* t = to + int64_t(le) * EF + f * NV * NF + q;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      FxAcc a{0, 0};
#pragma unroll
      for (int j = 0; j < NP; ++j) fx_mac(a, sv[pts[j] + v * N], c[j]);
      const uint32_t e = se[le * FX_GROUPS + fx_group(v, NV)];
      t[v * NF] = fx_double(fx_sum(a), fx_unit(fx_exp(e), kt), e >= FX_E_BAD);
    }
  }
}
// Then, in a block that has some, the traces of the elements of wide range (wide[le], see fx_low) again, as FP64
// chains from the state u in memory, each by the thread that wrote the first one.  With one exponent per
// group and element the thin side of a jump r inside an element has traces off by 2^-59 r of themselves; the
// wave speeds formed from them carried that into the whole residual (1e-13 of it at r = 1e5, 1e-10 at 1e8,
// now 5e-16).  Rare, so not inlined, and with the operator's entries from the fixed-point ones, into sl[2 NP]
// (tables of their own among the kernel's parameters cost every launch 0.3 us).  All threads of the block.
template <int DIM, int NP>
__device__ __noinline__ void wide_traces(const double* u, const int2* slm, const int2* slp, int kt, double* sl,
                                         int ne, const int8_t* wide, const int8_t* need, double* to) {
  using S = Sz<DIM, NP>;
  constexpr int N = S::N, NV = S::NV, NF = S::NF, EU = S::EU, EF = S::EF, FQ = S::NFC * NF;
  if (threadIdx.x < 2 * NP)
    sl[threadIdx.x] = fx_coef_value(threadIdx.x < NP ? slm[threadIdx.x] : slp[threadIdx.x - NP], kt);
  __syncthreads();
  for (int k = threadIdx.x; k < ne * FQ; k += blockDim.x) {
    const int le = k / FQ, r = k % FQ, f = r / NF, q = r % NF;
    if (!wide[le] || (need && !need[le])) continue;
    const double* l = sl + (f & 1) * NP;
    for (int v = 0; v < NV; ++v) {
      double t = 0.0;
#pragma unroll
      for (int j = 0; j < NP; ++j) t = fma(l[j], u[le * EU + v * N + line_pt<DIM, NP>(f >> 1, q, j)], t);
      to[int64_t(le) * EF + (f * NV + v) * NF + q] = t;
    }
  }
}

// traces tr[e][f][v][q] = sum_j l_j(+-1) u[e][v][line point j] of a whole mesh, bitwise those that the
// element kernel writes with a state (blocks of EPB elements, one thread per point)
template <int DIM, int NP>
__global__ void __launch_bounds__(Sz<DIM, NP>::BT) k_traces_fx(const double* __restrict__ u, int64_t M,
                                                               const __grid_constant__ TraceFx ops,
                                                               double* __restrict__ tr,
                                                               const int8_t* __restrict__ mask,
                                                               const int64_t* __restrict__ d_M) {
  pdl_wait_then_release();
  using S = Sz<DIM, NP>;
  constexpr int N = S::N, NV = S::NV, EU = S::EU, EPB = S::EPB;
  __shared__ int2 sv[EPB * EU];
  __shared__ int2 slm[NP], slp[NP];
  __shared__ uint32_t se[EPB * FX_GROUPS];
  __shared__ int8_t need[EPB], wide[EPB];
  __shared__ int low;
  __shared__ double sl[2 * NP];
  const int tid = threadIdx.x;
  if (d_M && *d_M < M) M = *d_M;  // the element count on the device (M is then a bound of it)
  const int64_t e0 = int64_t(blockIdx.x) * EPB;
  if (e0 >= M) return;
  const int ne = int((M - e0) < EPB ? (M - e0) : EPB);
  const int le = tid / N, i = tid % N;
  if (tid < ne) {
    need[tid] = mask ? mask[e0 + tid] : 1;
    wide[tid] = 0;
  }
  if (tid == 0) low = 0;
  if (tid < NP) {
    slm[tid] = ops.lm[tid];
    slp[tid] = ops.lp[tid];
  }
  for (int k = tid; k < EPB * FX_GROUPS; k += blockDim.x) se[k] = 0u;
  __syncthreads();
  const bool act = le < ne && need[le < EPB ? le : 0];
  double q[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) q[v] = act ? u[(e0 + le) * EU + v * N + i] : 0.0;
  uint32_t w[FX_GROUPS] = {0u, 0u, 0u};
  if (act) fx_state_exps<NV>(q, w);
  fx_group_max<N>(w, i, act, se + (act ? le : 0) * FX_GROUPS);
  __syncthreads();
  if (act) {
    if (fx_low_state(w, se + le * FX_GROUPS)) wide[le] = low = 1;
#pragma unroll
    for (int v = 0; v < NV; ++v)
      sv[le * EU + v * N + fx_place<DIM, NP>(i)] = fx_limbs(q[v], fx_exp(se[le * FX_GROUPS + fx_group(v, NV)]));
  }
  __syncthreads();
  fx_traces<DIM, NP>(sv, se, slm, slp, ops.kt, ne, need, tr + e0 * S::EF);
  if (low) wide_traces<DIM, NP>(u + e0 * EU, slm, slp, ops.kt, sl, ne, wide, need, tr + e0 * S::EF);
}

// planes of the element's fluxes: the axes' mass fluxes, the distinct entries of the symmetric
// momentum flux tensor, the axes' energy fluxes
template <int DIM>
struct FluxPlanes {
  static constexpr int NS = DIM * (DIM + 1) / 2;
  static constexpr int NPL = 2 * DIM + NS;
  // row a, column b of the symmetric tensor
  static __host__ __device__ constexpr int sym(int a, int b) {
    return (a < b ? a : b) * DIM - (a < b ? a : b) * ((a < b ? a : b) - 1) / 2 + (a < b ? b - a : a - b);
  }
  // exponent group of plane k
  static __host__ __device__ constexpr int group(int k) { return k < DIM ? 0 : (k < DIM + NS ? 1 : 2); }
  // plane of variable v's flux along axis a
  static __host__ __device__ constexpr int of(int a, int v) {
    return v == 0 ? a : (v == DIM + 1 ? DIM + NS + a : DIM + sym(a, v - 1));
  }
};

// Resident blocks the element kernel is compiled for.  It waits on shared memory, barriers and fixed
// latencies more than on any one pipe, so threads are worth more than registers: 1024 threads an SM (64
// registers, a few spilled) against 768 and 512 give, per launch, 3D p = 2 (184k leaves) 587, 631 and 712
// us, 3D p = 4 (15k) 230, 242 and 258 us; at 3D p = 3 (127k), 896 threads are best: 838 us against 853
// (1024), 872 (768) and 903 (640).  Blocks of 64 threads instead of 128: 894 us.
template <int DIM, int NP>
struct StageOcc {
  static constexpr int value = (Sz<DIM, NP>::N == 64 ? 896 : 1024) / Sz<DIM, NP>::BT;
};

// Element stage of the FP64 form: R = -sum_a (2/h) [ sum_j Dt_ij f_j + gL_i F(-1) + gR_i F(+1) ]
// along each axis (corrected-flux derivative of Sec. 2.1 with the correction folded into Dt; the
// interface kernel stores 2F and the slopes carry the 1/2), then out = a*un + b*us + c*R (Eq. rk3)
// and (optionally) the flags of out and its traces.
//
// The pointwise flux and the Runge-Kutta combination are FP64 (36 operations a point in 3D, 26 in the first
// stage, of the 158 that bounded the kernel at 2 a clock and SM); the contractions run in fixed point on the
// integer pipes (fr_fixed.cuh), all axes of a variable in one accumulator, the correction's terms in the
// derivative's accumulator once that has moved to the larger of the two exponents, so that the volume part
// stays before the wait on the interface kernel.  Per point about 2,400 instructions (a third of them the
// conversions of 28 values to limbs and 13 back); FP64 pipe 55%, issue slots 54%, shared memory 59% busy,
// DRAM 28% of peak.  Four 3D p = 3 tubes, 127k leaves: 2166 us per launch with the contractions in FP64,
// 825 us so (838 without the spread places of fx_place and u^n's prefetch).
//
// Elements of wide range (fx_low) take FP64 chains.  A point that is too low sets a flag of its block before a
// barrier that the block has anyway, and the block leaves for a body of its own that is not inlined.  Per
// launch at 3D p = 3 with 242k leaves: 1597 us without the test, 1703 with branches inside or with a vote by
// the barrier (__syncthreads_or), 1597 so (3D p = 2, 184k: 603, 620 and 603 us; 2D p = 3, 11k: 21.9 and 22.6 us).
// Blocks that do leave take about three times as long, 20 to 32% longer than when the whole form was FP64.
template <int DIM, int NP>
struct StageMem {
  using S = Sz<DIM, NP>;
  static constexpr int EPB = S::EPB;
  int2 fl[EPB * FluxPlanes<DIM>::NPL * S::N];  // fluxes; after the derivative the new state
  int2 fc[EPB * S::EF];                        // common fluxes
  int2 D[NP * NP], gL[NP], gR[NP], lm[NP], lp[NP];
  uint32_t ef[EPB * FX_GROUPS], ec[EPB * FX_GROUPS], eo[EPB * FX_GROUPS];  // exponents: fluxes, common fluxes, new state
  uint32_t rho0[EPB];           // exponent of the first point's density
  int low[2];                   // a point too low for its element's exponents: old state, new state
  int8_t wide[EPB];             // elements of wide range (mixed body)
  double f64[NP * NP + 2 * NP];  // their operators' entries: D, gL, gR; then l(-1), l(+1)
  double h2[EPB];               // per element: c * (-2/h)
  unsigned long long g2[EPB];   // per element: the indicator's max |D rho|^2 (as bits)
};

// Traces of a block's elements of wide range, from the new state in memory
template <int DIM, int NP>
__device__ __noinline__ void stage_traces_wide(const StageArgs& A, const OpsFx& ops, StageMem<DIM, NP>& m) {
  using S = Sz<DIM, NP>;
  constexpr int N = S::N, NV = S::NV, EU = S::EU;
  const int tid = threadIdx.x, le = tid / N;
  const int64_t e0 = int64_t(blockIdx.x) * S::EPB;
  const int ne = int((A.M - e0) < S::EPB ? (A.M - e0) : S::EPB);
  const double* u = A.out + e0 * EU;
  if (tid < ne) m.wide[tid] = 0;
  __syncthreads();
  if (le < ne) {
    double q[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = u[le * EU + v * N + tid % N];
    uint32_t w[FX_GROUPS];
    fx_state_exps<NV>(q, w);
    if (fx_low_state(w, m.eo + le * FX_GROUPS)) m.wide[le] = 1;
  }
  __syncthreads();
  wide_traces<DIM, NP>(u, m.lm, m.lp, ops.tr.kt, m.f64, ne, m.wide, nullptr,
                       static_cast<double*>(A.trace_out) + e0 * S::EF);
}

// The element stage from the derivative on (fluxes staged, exponents known)
template <int DIM, int NP, bool MIXED>
__device__ __forceinline__ void stage_rest(const StageArgs& A, const OpsFx& ops, StageMem<DIM, NP>& m,
                                           int (&E)[FX_GROUPS]) {
  using S = Sz<DIM, NP>;
  using FP = FluxPlanes<DIM>;
  constexpr int N = S::N, NV = S::NV, NF = S::NF, EU = S::EU, EF = S::EF, EPB = S::EPB, BT = S::BT, NPL = FP::NPL;
  constexpr int FQ = S::NFC * NF, NIT = (EPB * FQ + BT - 1) / BT;
  const int tid = threadIdx.x;
  const int64_t e0 = int64_t(blockIdx.x) * EPB;
  const int ne = int((A.M - e0) < EPB ? (A.M - e0) : EPB);
  const int i = tid % N;
  const bool own = EPB * N == BT || tid < EPB * N;
  const int le = own ? tid / N : 0;
  const bool act = own && le < ne;
  const int64_t b0 = (e0 + (le < ne ? le : ne - 1)) * EU + i;
  const bool wide = MIXED && m.wide[le];  // this thread's element in FP64
  // volume part of the folded derivative, sum_a sum_j Dt_ij f_j
  FxAcc acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = FxAcc{0, 0};
  double vol[NV];
  if (MIXED && wide) {
#pragma unroll
    for (int v = 0; v < NV; ++v) vol[v] = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      int qf, ia;
      pt_split<DIM, NP>(i, a, &qf, &ia);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const double* f = reinterpret_cast<const double*>(m.fl) + le * NPL * N + line_pt<DIM, NP>(a, qf, j);
        const double d = m.f64[ia * NP + j];
#pragma unroll
        for (int v = 0; v < NV; ++v) vol[v] = fma(d, f[FP::of(a, v) * N], vol[v]);
      }
    }
  } else {
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      int qf, ia;
      pt_split<DIM, NP>(i, a, &qf, &ia);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const int2 c = m.D[ia * NP + j];
        const int2* f = m.fl + le * NPL * N + line_pt<DIM, NP>(a, qf, j);
#pragma unroll
        for (int v = 0; v < NV; ++v) fx_mac(acc[v], f[FP::of(a, v) * N], c);
      }
    }
  }
  pdl_wait_then_release();
  // common fluxes of the block's elements, one thread per face point: staged in FP64 while the group
  // exponents are formed, then converted in place
#pragma unroll
  for (int t = 0; t < NIT; ++t) {
    const int k = tid + t * BT;
    const bool in = (t + 1) * BT <= EPB * FQ || k < EPB * FQ;
    if ((EPB * FQ) % 32 == 0 && FQ % 32 == 0 && !in) break;  // whole warps
    const int lf = in ? k / FQ : 0, r = k % FQ, o = (r / NF) * NV * NF + r % NF;
    const double* fc = static_cast<const double*>(A.fcomm) + (e0 + (lf < ne ? lf : ne - 1)) * EF + o;
    uint32_t w[FX_GROUPS] = {0u, 0u, 0u};
    if (in) {
      double F[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) F[v] = fc[v * NF];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        w[fx_group(v, NV)] = max(w[fx_group(v, NV)], fx_mag(F[v]) >> 20);
        reinterpret_cast<double*>(m.fc)[lf * EF + o + v * NF] = F[v];
      }
    }
    fx_group_max<FQ>(w, r, in, m.ec + lf * FX_GROUPS);
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < NIT; ++t) {
    const int k = tid + t * BT;
    if ((t + 1) * BT <= EPB * FQ || k < EPB * FQ) {
      const int lf = k / FQ, r = k % FQ, o = lf * EF + (r / NF) * NV * NF + r % NF;
      int Ec[FX_GROUPS];
#pragma unroll
      for (int g = 0; g < FX_GROUPS; ++g)
        Ec[g] = fx_exp(max(m.ef[lf * FX_GROUPS + g], m.ec[lf * FX_GROUPS + g]));
#pragma unroll
      for (int v = 0; v < NV; ++v)
        m.fc[o + v * NF] = fx_limbs(reinterpret_cast<const double*>(m.fc)[o + v * NF], Ec[fx_group(v, NV)]);
    }
  }
  // the sums move to the larger exponent of fluxes and common fluxes
  {
    int sh[FX_GROUPS];
#pragma unroll
    for (int g = 0; g < FX_GROUPS; ++g) {
      const int Ec = max(E[g], fx_exp(m.ec[le * FX_GROUPS + g]));
      sh[g] = min(Ec - E[g], 63);
      E[g] = Ec;
    }
    if (sh[0] | sh[1] | sh[2]) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (sh[fx_group(v, NV)]) acc[v] = FxAcc{fx_sum(acc[v]) >> sh[fx_group(v, NV)], 0};
    }
  }
  __syncthreads();
  double out[NV];
  {
    // u_s and u^n of the combination, read here (u_s from the caches) to keep the registers free
    double unr[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      out[v] = A.us[b0 + v * N];
      if (A.rk & RK_A) unr[v] = A.un[b0 + v * N];
    }
    const double* F = static_cast<const double*>(A.fcomm) + (e0 + (le < ne ? le : ne - 1)) * EF;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      int qf, ia;
      pt_split<DIM, NP>(i, a, &qf, &ia);
      const int2 cl = m.gL[ia], cr = m.gR[ia];
      const int2* Fm = m.fc + le * EF + (2 * a) * NV * NF + qf;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        fx_mac(acc[v], Fm[v * NF], cl);
        fx_mac(acc[v], Fm[(NV + v) * NF], cr);
      }
      if (MIXED && wide) {
        const double dl = m.f64[NP * NP + ia], dr = m.f64[NP * NP + NP + ia];
#pragma unroll
        for (int v = 0; v < NV; ++v)
          vol[v] = fma(dl, F[(2 * a * NV + v) * NF + qf], fma(dr, F[((2 * a + 1) * NV + v) * NF + qf], vol[v]));
      }
    }
    const double cs = m.h2[le < ne ? le : 0];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int Ev = E[fx_group(v, NV)];
      double R = fx_double(fx_sum(acc[v]), fx_unit(Ev, ops.kd), Ev >= FX_E_BAD);
      if (MIXED && wide) R = vol[v];
      // the first stage (a = 0, b = 1) is one FMA per value; the tests are uniform over the grid
      double o = fma(cs, R, (A.rk & RK_B1) ? out[v] : A.b * out[v]);
      if (A.rk & RK_A) o = fma(A.a, unr[v], o);
      out[v] = o;
    }
  }
  if (act) {
#pragma unroll
    for (int v = 0; v < NV; ++v) A.out[b0 + v * N] = out[v];
  }
  if (A.flags) {
    // the density-gradient indicator of the new state (the same arithmetic as the indicator
    // kernel): eta = 2 max_i |D_xi rho|, flags from the thresholds
    double* rho = reinterpret_cast<double*>(m.fl) + le * N;
    if (act) rho[i] = out[0];
    __syncthreads();
    if (act) {
      double g2 = 0.0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        int qf, ia;
        pt_split<DIM, NP>(i, a, &qf, &ia);
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < NP; ++j) d += ops.D[ia][j] * rho[line_pt<DIM, NP>(a, qf, j)];
        g2 += d * d;
      }
      atomicMax(&m.g2[le], static_cast<unsigned long long>(__double_as_longlong(g2)));  // g2 >= 0
    }
    __syncthreads();
    if (act && i == 0) {
      const double val = 2.0 * sqrt(__longlong_as_double(static_cast<long long>(m.g2[le])));
      A.flags[e0 + le] = int8_t(val > A.th_r ? 1 : (val < A.th_c ? -1 : 0));
    }
  }
  if (A.trace_out) {
    uint32_t w[FX_GROUPS];
    fx_state_exps<NV>(out, w);
    if (!own) w[0] = w[1] = w[2] = 0u;
    fx_group_max<N>(w, i, own, m.eo + le * FX_GROUPS);
    __syncthreads();
    const uint32_t* se = m.eo + le * FX_GROUPS;
    const uint32_t e[FX_GROUPS] = {se[0], se[1], se[2]};
    if (own) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        m.fl[le * EU + v * N + fx_place<DIM, NP>(i)] = fx_limbs(out[v], fx_exp(e[fx_group(v, NV)]));
    }
    if (act && fx_low_state(w, e)) m.low[1] = 1;
    __syncthreads();
    fx_traces<DIM, NP>(m.fl, m.eo, m.lm, m.lp, ops.tr.kt, ne, nullptr, static_cast<double*>(A.trace_out) + e0 * EF);
    if (m.low[1]) stage_traces_wide<DIM, NP>(A, ops, m);
  }
}
// a point whose momentum fluxes, which hold the pressure, are too low for the element's exponents ef, or
// whose density is more than half of FX_SPREAD exponents from the first point's (which takes no reduction)
__device__ __forceinline__ bool stage_low(uint32_t e_mom, uint32_t e_rho, const uint32_t* ef, uint32_t rho0) {
  return fx_low(e_mom, ef[1]) || e_rho + FX_SPREAD / 2 - rho0 > uint32_t(FX_SPREAD) - 1u;
}
template <int DIM>
__device__ __forceinline__ void point_fluxes(const double* q, double gm1, double ngmh, double* fl) {
  using FP = FluxPlanes<DIM>;
  constexpr int NV = DIM + 2;
  const double rinv = rcp_t(q[0]);
  double vel[DIM];
  double m2 = 0.0;
#pragma unroll
  for (int b = 0; b < DIM; ++b) {
    vel[b] = q[1 + b] * rinv;
    m2 = b == 0 ? q[1] * vel[0] : fma(q[1 + b], vel[b], m2);
  }
  const double p = fma(ngmh, m2, gm1 * q[NV - 1]);
  const double Ep = q[NV - 1] + p;
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    fl[FP::of(a, 0)] = q[1 + a];
#pragma unroll
    for (int b = a; b < DIM; ++b) fl[FP::of(a, 1 + b)] = a == b ? fma(q[1 + b], vel[a], p) : q[1 + b] * vel[a];
    fl[FP::of(a, NV - 1)] = Ep * vel[a];
  }
}
// exponents of a point's fluxes
template <int DIM>
__device__ __forceinline__ void flux_exps(const double* fl, uint32_t (&w)[FX_GROUPS]) {
  using FP = FluxPlanes<DIM>;
  w[0] = w[1] = w[2] = 0u;
#pragma unroll
  for (int k = 0; k < FP::NPL; ++k) w[FP::group(k)] = max(w[FP::group(k)], fx_mag(fl[k]));
#pragma unroll
  for (int g = 0; g < FX_GROUPS; ++g) w[g] >>= 20;
}
// The rest of a block with elements of wide range: their fluxes take the limbs' places as doubles
template <int DIM, int NP>
__device__ __noinline__ void stage_rest_mixed(const StageArgs& A, const OpsFx& ops, StageMem<DIM, NP>& m) {
  using S = Sz<DIM, NP>;
  constexpr int N = S::N, NV = S::NV, EU = S::EU, EPB = S::EPB, NPL = FluxPlanes<DIM>::NPL;
  const int tid = threadIdx.x, i = tid % N, le = tid / N;
  const int64_t e0 = int64_t(blockIdx.x) * EPB;
  const int ne = int((A.M - e0) < EPB ? (A.M - e0) : EPB);
  if (tid < EPB) m.wide[tid] = 0;
  if (tid < NP * NP + 2 * NP)
    m.f64[tid] = fx_coef_value(
        tid < NP * NP ? m.D[tid] : (tid < NP * NP + NP ? m.gL[tid - NP * NP] : m.gR[tid - NP * NP - NP]), ops.kd);
  __syncthreads();
  double fl[NPL];
  if (le < ne) {
    double q[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = A.us[(e0 + le) * EU + v * N + i];
    point_fluxes<DIM>(q, ops.gm1, ops.ngmh, fl);
    uint32_t w[FX_GROUPS];
    flux_exps<DIM>(fl, w);
    if (stage_low(w[1], fx_mag(q[0]) >> 20, m.ef + le * FX_GROUPS, m.rho0[le])) m.wide[le] = 1;
  }
  __syncthreads();
  if (le < ne && m.wide[le]) {
#pragma unroll
    for (int k = 0; k < NPL; ++k) reinterpret_cast<double*>(m.fl)[(le * NPL + k) * N + i] = fl[k];
  }
  __syncthreads();
  int E[FX_GROUPS];
#pragma unroll
  for (int g = 0; g < FX_GROUPS; ++g) E[g] = fx_exp(m.ef[(EPB * N == S::BT || tid < EPB * N ? le : 0) * FX_GROUPS + g]);
  stage_rest<DIM, NP, true>(A, ops, m, E);
}

template <int DIM, int NP>
__global__ void __launch_bounds__(Sz<DIM, NP>::BT, StageOcc<DIM, NP>::value)
    k_stage_fx(const __grid_constant__ StageArgs A, const __grid_constant__ OpsFx ops) {
  using S = Sz<DIM, NP>;
  using FP = FluxPlanes<DIM>;
  constexpr int N = S::N, NV = S::NV, EU = S::EU, EPB = S::EPB, BT = S::BT, NPL = FP::NPL;
  __shared__ StageMem<DIM, NP> m;
  const int tid = threadIdx.x;
  const int64_t e0 = int64_t(blockIdx.x) * EPB;
  const int ne = int((A.M - e0) < EPB ? (A.M - e0) : EPB);
  // threads past the last element repeat its work without storing it, threads past the last point
  // of the block (27, 9, 25 or 125 points an element) the first element's
  const int i = tid % N;
  const bool own = EPB * N == BT || tid < EPB * N;
  const int le = own ? tid / N : 0;
  const int64_t b0 = (e0 + (le < ne ? le : ne - 1)) * EU + i;
  // the stage's input state, the state at the start of the step and the keys come from earlier
  // launches than the interface kernel this one depends on: everything up to the volume sums is done
  // while that kernel drains; its common fluxes are read after the wait
  double q[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) q[v] = A.us[b0 + v * N];
  // u^n is read at the end: into the second-level cache meanwhile
  if (A.rk & RK_A)
    for (int k = tid * 16; k < ne * EU; k += BT * 16)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(A.un + e0 * EU + k));
  // c * (-2/h): 2^depth * (2/L) is exact, so this equals the rounded -2^(depth+1)/L times c
  if (tid < ne) {
    m.h2[tid] = -A.c * (double(1ull << A.g.depth(A.keys[e0 + tid])) * A.twoL);
    m.g2[tid] = 0ull;
  }
  if (tid < 2) m.low[tid] = 0;
  for (int k = tid; k < EPB * FX_GROUPS; k += BT) m.ef[k] = m.ec[k] = m.eo[k] = 0u;
  for (int k = tid; k < NP * NP; k += BT) m.D[k] = ops.Dt[k / NP][k % NP];
  if (tid < NP) {
    m.gL[tid] = ops.gLh[tid];
    m.gR[tid] = ops.gRh[tid];
    m.lm[tid] = ops.tr.lm[tid];
    m.lp[tid] = ops.tr.lp[tid];
  }
  __syncthreads();
  int E[FX_GROUPS];
  {
    // pointwise fluxes, FP64
    double fl[NPL];
    point_fluxes<DIM>(q, ops.gm1, ops.ngmh, fl);
    uint32_t w[FX_GROUPS];
    flux_exps<DIM>(fl, w);
    if (!own) w[0] = w[1] = w[2] = 0u;
    fx_group_max<N>(w, i, own, m.ef + le * FX_GROUPS);
    const uint32_t e_rho = fx_mag(q[0]) >> 20;
    // the element's first density: by a shuffle where elements lie in a warp (the mixed body reads it, too)
    uint32_t rho0 = 32 % N == 0 ? __shfl_sync(~0u, e_rho, (tid & 31) / N * N) : 0u;
    if (own && i == 0) m.rho0[le] = e_rho;
    __syncthreads();
    if (32 % N != 0) rho0 = m.rho0[le];
    const uint32_t* se = m.ef + le * FX_GROUPS;
    const uint32_t e[FX_GROUPS] = {se[0], se[1], se[2]};
    const bool low = own && stage_low(w[1], e_rho, e, rho0);
#pragma unroll
    for (int g = 0; g < FX_GROUPS; ++g) E[g] = fx_exp(e[g]);
    if (own) {
#pragma unroll
      for (int k = 0; k < NPL; ++k) m.fl[(le * NPL + k) * N + i] = fx_limbs(fl[k], E[FP::group(k)]);
    }
    if (low) m.low[0] = 1;
  }
  __syncthreads();
  if (!m.low[0]) {
    stage_rest<DIM, NP, false>(A, ops, m, E);
    return;
  }
  stage_rest_mixed<DIM, NP>(A, ops, m);
}

}  // namespace frg
