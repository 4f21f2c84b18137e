// Shared pieces of the formal-solution kernels: the evaluation mode of a
// column and the piecewise-linear coefficients of App. A.1 in the form the
// difference recurrences use.
#pragma once

#include "internal.cuh"

namespace jfnk {

__device__ __forceinline__ int eval_mode_f(const ColDesc& cd) {
  if (cd.forced_mode >= 0) return cd.forced_mode;
  switch (cd.w.st->phase) {
    case PH_BASE: return EV_BASE;
    case PH_JVP:
    case PH_RESTART: return cd.w.st->fd_scheme ? EV_FD : EV_TANGENT;
    case PH_RH92: return EV_RH92;
    default: return EV_SKIP;
  }
}

// First part slot of transition t in ColWork::rpart and its number of tiles,
// for the lane's transition (warp-wide; lanes past nt get 0).
__device__ __forceinline__ int part_offset(const ColTables& T, int qb, int lane, int& tile0, int& ntile) {
  tile0 = ntile = 0;
  if (lane < T.nt) {
    tile0 = T.t_q0[lane] / qb;
    ntile = T.t_q1[lane] / qb - tile0 + 1;
  }
  int s = ntile;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += v;
  }
  return s - ntile;
}

// Coefficients of one step of optical depth x: e = exp(-x), w = (1 - e)/x,
// a = 1 - w and bq = (w - e)/x, each from its own Taylor series below
// x = 0.1 (where 1 - e, 1 - w and w - e cancel); r = 1/x is supplied by the
// caller (shared between the rays of a layer).
// FP64 Taylor coefficients: w = sum_{n>=0} (-x)^n/(n+1)!,
// a/x = sum_{n>=0} (-x)^n/(n+2)!, bq = sum_{n>=0} (-x)^n (n+1)/(n+2)!.
__device__ __forceinline__ void pl_series64(double x, double& w, double& a, double& bq) {
  // terms up to n = 5: below x = 1e-3 the first omitted one is < 3e-23 relative
  constexpr double f[8] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040};
  double pw = 0.0, pa = 0.0, pb = 0.0;
#pragma unroll
  for (int m = 5; m >= 0; --m) {
    const double sg = (m & 1) ? -1.0 : 1.0;
    pw = fma(pw, x, sg * f[m + 1]);
    pa = fma(pa, x, sg * f[m + 2]);
    pb = fma(pb, x, sg * (m + 1) * f[m + 2]);
  }
  w = pw;
  a = pa * x;
  bq = pb;
}

// In FP64 the direct forms of w, a and bq lose about 1e-16/x^2 relative
// (1 - e, 1 - w and w - e cancel): 2e-10 at |x| = 1e-3, so the series takes
// over below |x| = 1e-3 only (x < 0: inverted populations).
__device__ __forceinline__ void pl_coef_f(double x, double r, double& e, double& w, double& a, double& bq) {
  e = exp(-x);
  if (fabs(x) < 1e-3) {
    pl_series64(x, w, a, bq);
  } else {
    w = (1.0 - e) * r;
    a = 1.0 - w;
    bq = (w - e) * r;
  }
}

__device__ __forceinline__ void pl_coef_f(float x, float r, float& e, float& w, float& a, float& bq) {
  e = __expf(-x);
  if (x < 0.1f) {
    w = fmaf(fmaf(fmaf(fmaf(fmaf(-1.0f / 720.0f, x, 1.0f / 120.0f), x, -1.0f / 24.0f), x, 1.0f / 6.0f), x, -0.5f), x, 1.0f);
    a = x * fmaf(fmaf(fmaf(fmaf(fmaf(-1.0f / 5040.0f, x, 1.0f / 720.0f), x, -1.0f / 120.0f), x, 1.0f / 24.0f), x, -1.0f / 6.0f), x, 0.5f);
    bq = fmaf(fmaf(fmaf(fmaf(1.0f / 144.0f, x, -1.0f / 30.0f), x, 1.0f / 8.0f), x, -1.0f / 3.0f), x, 0.5f);
  } else {
    w = (1.0f - e) * r;
    a = 1.0f - w;
    bq = (w - e) * r;
  }
}

// Every operation of a ray step is an explicitly rounded intrinsic: the
// compiler may not contract or reorder any of them, so the two kernel
// variants below (which see the same values in different registers, lanes
// and orders of issue) produce bit-identical results.
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fma3(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// Tangent of the opacity and source function at (nu, k) in FP32 (Eqs. chi,
// eta differentiated; n and J^dagger fixed): per active transition
//   dchi += V (dn_lo - g dn_up),  deta += g V dn_up   (eta normalised by 2 h nu^3/c^2)
// and dS = (deta - S dchi)/chi. Shared by the opacity kernel and the sweeps
// that form it on the fly, so that both give the same bits.
struct TanAcc {
  float dchi = 0.f, deta = 0.f;
};
__device__ __forceinline__ void tan_acc(TanAcc& t, float V, float g, float vlo, float vup) {
  t.dchi = fma3(V, sub(vlo, mul(g, vup)), t.dchi);
  t.deta = fma3(mul(g, V), vup, t.deta);
}
// Opacity and source function at (nu, k) of a mixed-mode base or RH92
// evaluation (Eqs. chi, eta): chi is stored in float, S (and the RH92
// emissivity) as float pairs; every sum runs in pair arithmetic on the FP32
// pipe (GB300's FP64 pipe is 1/64 of it): chi = chi_c + chi_sca + sum V n_lo -
// sum g V n_up, eta / (2 h nu^3/c^2) = (eta_c + chi_sca J^dagger) c^2/(2 h nu^3)
// + sum g V n_up; i = q nz + k.
struct BasePoint {
  float chi;
  df S;
};
// EARLY: the loads of the first three transitions are issued together (small
// launches, bound by latency; a large one is faster with fewer registers).
template <bool EARLY>
__device__ __forceinline__ BasePoint base_opacity(const ColDesc& cd, int mode, int q, int k, int i) {
  const ColTables& T = cd.t;
  const int nz = T.nz;
  const float2* n2 = cd.w.n2 + k * T.nl;
  const df jd = df_load(as_pairs(jdag_ptr(cd)), i);
  const df eta_bg = df_add(df_load(T.etac2, i), df_mul(df_load(T.chisca2, k), jd));
  df chl = df_make(0.f, 0.f), el = df_make(0.f, 0.f);
  if (EARLY && T.max_overlap <= kQMetaT) {
    constexpr int E = 3;
    const int4 a = __ldg(T.qmeta4 + 2 * (size_t)q), b = __ldg(T.qmeta4 + 2 * (size_t)q + 1);
    const int ms[kQMetaT] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    df V[E], gV[E], nl_[E], nu_[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int m = max(ms[j], 0);
      const size_t p = (size_t)(m >> 8) * nz + k;
      V[j] = df_load(T.V2, p);
      gV[j] = df_load(T.gV2, p);
      nl_[j] = df_load(n2, (m >> 4) & 15);
      nu_[j] = df_load(n2, m & 15);
    }
#pragma unroll
    for (int j = 0; j < kQMetaT; ++j) {
      const int m = ms[j];
      if (m < 0) break;
      if (j < E) {
        chl = df_add(chl, df_mul(V[j], nl_[j]));
        el = df_add(el, df_mul(gV[j], nu_[j]));
      } else {
        const size_t p = (size_t)(m >> 8) * nz + k;
        chl = df_add(chl, df_mul(df_load(T.V2, p), df_load(n2, (m >> 4) & 15)));
        el = df_add(el, df_mul(df_load(T.gV2, p), df_load(n2, m & 15)));
      }
    }
  } else if (T.max_overlap <= kQMetaT) {
    // the packed table gives window point and levels in one load
#pragma unroll
    for (int j = 0; j < kQMetaT; ++j) {
      const int m = __ldg(T.qmeta + (size_t)j * T.nq + q);
      if (m < 0) break;
      const size_t p = (size_t)(m >> 8) * nz + k;
      chl = df_add(chl, df_mul(df_load(T.V2, p), df_load(n2, (m >> 4) & 15)));
      el = df_add(el, df_mul(df_load(T.gV2, p), df_load(n2, m & 15)));
    }
  } else {
    for (int s = T.q_off[q]; s < T.q_off[q + 1]; ++s) {
      const int t = T.q_t[s];
      const size_t p = (size_t)(T.t_base[t] + q - T.t_q0[t]) * nz + k;
      chl = df_add(chl, df_mul(df_load(T.V2, p), df_load(n2, T.t_lo[t])));
      el = df_add(el, df_mul(df_load(T.gV2, p), df_load(n2, T.t_up[t])));
    }
  }
  const df chi = df_sub(df_add(df_load(T.chibg2, i), chl), el);
  const df etan = df_add(df_mul(eta_bg, df_load(T.rc2p, q)), el);
  BasePoint p;
  p.chi = chi.hi;
  p.S = df_div(etan, chi);
  reinterpret_cast<float*>(cd.w.chi)[i] = p.chi;
  df_store(as_pairs(cd.w.S), i, p.S);
  if (mode == EV_RH92) {   // for the RH92 rate sums
    df_store(as_pairs(cd.w.eta), i, df_add(eta_bg, df_mul(el, df_load(T.c2p, q))));
    cd.w.etab32[i] = eta_bg.hi;
  }
  return p;
}

// Hardware reciprocal (1 ulp): a single instruction without a slow-path
// branch, so that loops around it stay one basic block the compiler can
// software-pipeline. Its arguments (opacity sums) are positive normal numbers.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float tan_dS(const TanAcc& t, float S, float chi) {
  return mul(sub(t.deta, mul(S, t.dchi)), rcp_approx(chi));
}

}  // namespace jfnk
