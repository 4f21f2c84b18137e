// Mixed-precision formal solution + ray sums, one thread per (frequency,
// column): the thread carries every angle of a hemisphere at once (n_mu
// independent recurrences, the instruction-level parallelism of the sweep)
// and walks the column twice.
//
//   down sweep (mu < 0 rays, top to bottom): the per-depth sums of the
//     hemisphere over its angles go to a scratch array laid out [k][q], so
//     that the threads of a warp (consecutive frequencies) write one
//     contiguous segment per depth;
//   up sweep (mu > 0 rays, bottom to top): the hemisphere's own sums are added
//     to the stored ones and the depth's outputs are written (J, J_new,
//     Lambda_chi, Lambda_eta in base evaluations, dJ in tangent ones).
//
// No per-ray value is stored anywhere: the coefficients of a step (App. A.1,
// App. A.2) are formed in registers right where the recurrence needs them,
// and the optical-depth reciprocal of a layer is shared by the angles.
//
// The recurrences are those of the fused kernel (Eqs. Iplus/Iminus in the
// difference form D = I - S, the tangent dD, and in base evaluations the
// intensity form I with the re-anchoring of D on I - S); only the order of
// the ray sums differs: each hemisphere is summed over its angles first and
// the two hemisphere sums are then added.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "formal_coef.cuh"

namespace jfnk {

constexpr int kSweepParts = 5;   // base: sum D, sum |D|, sum I, sum dI/dchi, sum dI/deta (x 1/2 w)

// Scratch of the down sweep: [kSweepParts][nz][col_pitch(nq)] floats.
__host__ __device__ inline int sweep_pitch(int nq) { return col_pitch(nq); }

size_t sweep_scratch_bytes(int nq, int nz) {
  return sizeof(float) * (size_t)kSweepParts * nz * sweep_pitch(nq);
}

// App. A.1 coefficients of a step of optical depth x (r = 1/x): e = exp(-x),
// w = (1 - e)/x, a = 1 - w, bq = (w - e)/x; below x = 0.1 each comes from its
// Taylor series (truncated after x^5, below 3e-10 relative).
// e^(-x) on the MUFU as 2^(-x log2 e) (flush-to-zero: e below 2^-126 is 0).
__device__ __forceinline__ float exp_neg(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(mul(x, -1.4426950408889634f)));
  return y;
}

// Asynchronous 4-byte copies global -> shared (each thread copies and later
// reads back only its own words, so waiting on its own copy groups suffices).
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Fused tangent sweep: the line-table entries of each depth are copied into a
// shared-memory ring kRing - 1 depths ahead of the recurrence; a stage holds
// per thread V, G, v_lo, v_up of the first two transitions and S.
constexpr int kRing = 4;
constexpr int kRingSlots = 9;
__host__ __device__ inline size_t ring_floats(int threads) { return (size_t)kRing * kRingSlots * threads; }

// Which form of the coefficients a step takes: chosen per step (CM_EITHER),
// or known for every angle of the depth (CM_SERIES: all steps below 0.1;
// CM_DIRECT: none), the same choice as CM_EITHER makes for each step.
// CM_SELECT forms both and selects: no branch, for launches bound by latency.
enum CoefMode { CM_EITHER = 0, CM_SERIES = 1, CM_DIRECT = 2, CM_SELECT = 3 };

// (Steps of inverted populations, x < 0, take the series, which is off by 2e-4 at
// x = -1; FP64 takes the direct forms there. With those here too, H I-like columns in
// which a line lases ended 1e-6 to 1e-3 elsewhere.)
template <int CM = CM_EITHER>
__device__ __forceinline__ void pl_coef_rn(float x, float r, float& e, float& w, float& a, float& bq) {
  e = exp_neg(x);
  if (CM == CM_SELECT) {
    float es, ws, as, bs, ed, wd, ad, bd;
    pl_coef_rn<CM_SERIES>(x, r, es, ws, as, bs);
    pl_coef_rn<CM_DIRECT>(x, r, ed, wd, ad, bd);
    const bool thin = x < 0.1f;
    w = thin ? ws : wd;
    a = thin ? as : ad;
    bq = thin ? bs : bd;
  } else if (CM == CM_SERIES || (CM == CM_EITHER && x < 0.1f)) {
    w = fma3(fma3(fma3(fma3(fma3(-1.0f / 720.0f, x, 1.0f / 120.0f), x, -1.0f / 24.0f), x, 1.0f / 6.0f), x, -0.5f), x, 1.0f);
    a = mul(x, fma3(fma3(fma3(fma3(fma3(-1.0f / 5040.0f, x, 1.0f / 720.0f), x, -1.0f / 120.0f), x, 1.0f / 24.0f), x, -1.0f / 6.0f), x, 0.5f));
    bq = fma3(fma3(fma3(fma3(1.0f / 144.0f, x, -1.0f / 30.0f), x, 1.0f / 8.0f), x, -1.0f / 3.0f), x, 0.5f);
  } else {
    w = mul(sub(1.0f, e), r);
    a = sub(1.0f, w);
    bq = mul(sub(w, e), r);
  }
}

// Quantities of one depth step shared by all angles of a hemisphere.
struct StepIn {
  float csum;    // chi^k + chi^u
  float rs;      // 1/(chi^k + chi^u)
  float dzk;     // |z_k - z_u|
  float idzk;    // 1/|z_k - z_u|
  float tz;      // |dz| (chi^k + chi^u):   dtau = tz / (2 mu)
  float rz;      // 1/(|dz| (chi^k + chi^u)): 1/dtau = rz 2 mu
  float dtz;     // |dz| (dchi^k + dchi^u): ddtau = dtz / (2 mu)
  float dSin;    // S^u - S^k (formed from the S pairs, then rounded)
  float S0, Su;  // S^k, S^u
  float rc0;     // 1/chi^k
  float dcs;     // dchi^k + dchi^u
  float ddSin;   // dS^u - dS^k
};

// Contributions of one ray to the sums of its depth, each already x 1/2 w_mu.
struct RayOut {
  float xD, xI, xx, xe, xd;
};

// One step of one ray into depth k from its upstream neighbour u:
//   D^k  = D^u e + w (S^u - S^k)                                  (D = I - S)
//   dD^k = dD^u e - ddtau (e D^u + bq (S^u - S^k)) + w (dS^u - dS^k)
//   I^k  = I^u e + a S^k + b S^u,  b = bq dtau                      (base)
//   dI^k/dchi^k = -(S^k/chi^k) a - h (S^u - S^k) bq - h e D^u,      (App. A.2)
//   dI^k/deta^k = a/chi^k,  h = |dz|/(2 mu), dtau = h (chi^k + chi^u)
// In base evaluations D is re-anchored on I - S whenever that is the
// better-conditioned value: D carries an absolute error of the order of the
// largest |D| met upstream (attenuated along the ray), I - S one of the order
// of |I| + |S|.
// The part of a step that depends on the opacities only (RayCoef) and the
// recurrence itself are separate, so that the warp variant can form the
// coefficients of several depths before it steps through them.
struct RayCoef {
  float e;        // exp(-dtau)
  float X;        // w (S^u - S^k)
  float Y;        // tangent: bq (S^u - S^k)          | base: bq
  float Z;        // tangent: w (dS^u - dS^k)         | base: a S^k + b S^u
  float t;        // tangent: ddtau                   | base: h
  float sa, xe;   // base: (S^k/chi^k) factor a and 1/2 w_mu a/chi^k
};
template <bool TAN, int CM = CM_EITHER>
__device__ __forceinline__ RayCoef ray_coef(const StepIn& in, float inv2mu, float two_mu, float hw) {
  RayCoef c;
  // the depth's factors are formed once per depth (StepIn), one multiply per angle here
  const float dtau = mul(in.tz, inv2mu);
  const float rdt = mul(in.rz, two_mu);
  float w, a, bq;
  pl_coef_rn<CM>(dtau, rdt, c.e, w, a, bq);
  c.X = mul(w, in.dSin);
  if (TAN) {
    c.t = mul(in.dtz, inv2mu);
    c.Y = mul(bq, in.dSin);
    c.Z = mul(w, in.ddSin);
    c.sa = c.xe = 0.f;
  } else {
    c.t = mul(in.dzk, inv2mu);
    c.Y = bq;
    c.Z = fma3(a, in.S0, mul(mul(bq, dtau), in.Su));
    c.sa = a;
    c.xe = mul(hw, mul(a, in.rc0));
  }
  return c;
}
template <bool TAN>
__device__ __forceinline__ RayOut ray_apply(const RayCoef& c, float dSin, float S0, float rc0, float hw, float& D,
                                            float& I, float& M, float& dD) {
  RayOut o;
  const float Du = D;
  float Dn = fma3(Du, c.e, c.X);
  if (TAN) {
    const float dDn = fma3(dD, c.e, fma3(-c.t, fma3(c.e, Du, c.Y), c.Z));
    dD = dDn;
    o.xd = mul(hw, dDn);
    o.xD = o.xI = o.xx = o.xe = 0.f;
  } else {
    const float In = fma3(I, c.e, c.Z);
    const float lx = -fma3(mul(S0, rc0), c.sa, mul(c.t, fma3(dSin, c.Y, mul(c.e, Du))));
    o.xI = mul(hw, In);
    o.xx = mul(hw, lx);
    o.xe = c.xe;
    M = fmaxf(mul(M, c.e), fabsf(Dn));
    const float anchor = add(fabsf(In), fabsf(S0));
    if (anchor < M) {
      Dn = sub(In, S0);
      M = anchor;
    }
    I = In;
    o.xD = mul(hw, Dn);
    o.xd = 0.f;
  }
  D = Dn;
  return o;
}
template <bool TAN, int CM = CM_EITHER>
__device__ __forceinline__ RayOut ray_step(const StepIn& in, float inv2mu, float two_mu, float hw, float& D,
                                           float& I, float& M, float& dD) {
  const RayCoef c = ray_coef<TAN, CM>(in, inv2mu, two_mu, hw);
  return ray_apply<TAN>(c, in.dSin, in.S0, in.rc0, hw, D, I, M, dD);
}

// Sum of the angle contributions in the fixed tree of a 3-level xor butterfly
// over 8 lanes, (x0 + x4) + (x2 + x6) and (x1 + x5) + (x3 + x7), with the terms
// of angles m >= MU (zero by construction, known at compile time) left out:
// x + 0 = x, so the sum has the butterfly's value.
struct Part {
  float v;
  bool on;
};
__device__ __forceinline__ Part padd(Part a, Part b) {
  if (a.on && b.on) return Part{add(a.v, b.v), true};
  return a.on ? a : b;
}
template <int MU>
__device__ __forceinline__ float tree_mu(const float* x) {
  Part p[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) p[i] = Part{i < MU ? x[i] : 0.f, i < MU};
  const Part s = padd(padd(padd(p[0], p[4]), padd(p[2], p[6])), padd(padd(p[1], p[5]), padd(p[3], p[7])));
  return s.on ? s.v : 0.f;
}
// Output of one depth from the two hemisphere sums (base: D, |D|, I, Lchi, Leta).
// J = (S + sum D) c2, or (sum I) c2 where that representation carries the
// smaller rounding error (intensities are >= 0), is formed in pair arithmetic
// and written once, into J_new (the rates read it there); the Lambda
// diagonals are FP32 sums and stay float. The sweeps serve the mixed mode
// only, whose Jacobian-vector products are exact tangents (no difference
// evaluations).
struct BaseOut {
  df J;
  float lx, le;
};
__device__ __forceinline__ BaseOut base_out(df Sk, df c2, float c2f, float fD, float fa, float fI, float fx, float fe) {
  BaseOut r;
  r.J = fabsf(fI) < fa ? df_mul_f(c2, fI) : df_mul(df_add_f(Sk, fD), c2);
  r.lx = mul(fx, c2f);
  r.le = fe;
  return r;
}
__device__ __forceinline__ void write_base(const ColDesc& cd, size_t o, df Sk, df c2, float c2f, float fD, float fa,
                                           float fI, float fx, float fe) {
  const BaseOut r = base_out(Sk, c2, c2f, fD, fa, fI, fx, fe);
  df_store(as_pairs(jnew_ptr(cd)), o, r.J);
  cd.w.Lchi32[o] = r.lx;
  cd.w.Leta32[o] = r.le;
}

// Outward pass of a base-type sweep: the per-frequency output rows ([q][k]:
// J pair, Lchi, Leta) are staged per warp for kStageD depths in shared memory
// ([plane][lane][depth], row stride kStageD + 1: the 32 lanes' words of one
// depth fall in 32 banks) and then written row by row, consecutive lanes on
// consecutive depths of a row, instead of one scattered word per lane.
// (Staging the input rows the same way, through a double buffer of
// asynchronous copies, was slower: 1.02 against 0.94 ms per tick; the larger
// shared memory leaves less L1, where those rows are mostly hits.)
constexpr int kStageD = 8;
constexpr int kStagePlane = 32 * (kStageD + 1);
constexpr int kWarpStage = 4 * kStagePlane;
__host__ __device__ inline size_t stage_floats(int threads) { return (size_t)(threads / 32) * kWarpStage; }
// Tangent output: dJ (normalised by 2 h nu^3/c^2) in float, depth-major, read
// by the FP32 tangent rate integrals; o indexes the depth-major arrays.
__device__ __forceinline__ void write_tan(const ColDesc& cd, size_t o, float dS, float fd) {
  cd.w.dJ32T[o] = add(dS, fd);
}

// Stages |dz| and 1/|dz| of the block's column in shared memory.
__device__ __forceinline__ void stage_dz(const ColTables& T, float* s_dz, float* s_idz) {
  for (int k = threadIdx.x; k < T.nz - 1; k += blockDim.x) {
    const float2 d = T.dz32[k];
    s_dz[k] = d.x;
    s_idz[k] = d.y;
  }
}

// ---------------------------------------------------------------------------
// Variant 1: one thread per frequency, all angles of a hemisphere in registers (the
// tangent sweep of a large launch: per two frequencies, sweep_pair below).
// ---------------------------------------------------------------------------
// Base evaluations read chi and S per frequency row ([q][k], S as a float
// pair), form S^u - S^k in pair arithmetic, and leave depth-major float
// copies of chi, S and the rounded differences for the tangent evaluations
// of the same Newton step;
// those then read depth-major float arrays only (one 128-byte line per warp
// and depth) and run entirely in FP32.
// EXACT: the column has exactly MU angles (no per-angle guards). FUSE
// (tangent, inward pass): the opacity tangent dchi, dS of each depth is formed
// here from the line tables, with the arithmetic of the separate opacity
// kernel (tan_acc, tan_dS: the same bits), and stored for the outward pass.
template <int MU, bool TAN, bool UP, bool EXACT, bool FUSE = false>
__device__ __forceinline__ void sweep_thread(const ColDesc& cd, int q, const float* __restrict__ s_dz,
                                             const float* __restrict__ s_idz, float* __restrict__ s_ring = nullptr,
                                             float* __restrict__ s_stage = nullptr, unsigned amask = 0u,
                                             int na = 0) {
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq, nmu = T.nmu, nl = T.nl;
  const size_t pitch = (size_t)col_pitch(nq);
  const size_t pstride = (size_t)nz * pitch;
  const size_t row = (size_t)q * nz;
  const float* __restrict__ chi = reinterpret_cast<const float*>(cd.w.chi) + row;
  const float2* __restrict__ S2 = as_pairs(cd.w.S) + row;   // S as float pairs
  float* __restrict__ chiT = cd.w.chiT + q;
  float* __restrict__ S32T = cd.w.S32T + q;
  float* __restrict__ dSkT = cd.w.dSkT + q;
  const float* __restrict__ dchiT = cd.w.dchiT + q;
  const float* __restrict__ dS32T = cd.w.dS32T + q;
  float* __restrict__ part = reinterpret_cast<float*>(cd.w.part) + q;
  const double c2 = T.c2[q];
  const float c2f = T.c2f[q];
  const df c2p = df_load(T.c2p, q);

  float inv2mu[MU], hw[MU], two_mu[MU];
#pragma unroll
  for (int m = 0; m < MU; ++m) {
    const bool on = EXACT || m < nmu;
    const float4 a = on ? T.ang32[m] : make_float4(0.f, 0.f, 0.f, 0.f);
    inv2mu[m] = a.x;
    hw[m] = a.y;
    two_mu[m] = a.z;
  }
  // the transitions active at nu (packed window point << 8 | lo << 4 | up),
  // constant along the column: the first two held, the others read when used
  constexpr bool FT = FUSE && TAN && !UP;
  int pm0 = -1, pm1 = -1;
  if (FT) {
    pm0 = __ldg(T.qmeta + q);
    pm1 = __ldg(T.qmeta + (size_t)nq + q);
  }
  // FUSE: the asynchronous copies of depth kk's table entries into ring stage
  // kk % kRing (one commit group per depth, empty past the column's end)
  const int bd = blockDim.x;
  auto tan_issue = [&](int kk) {
    if (kk < nz) {
      float* r = s_ring + (size_t)(kk % kRing) * kRingSlots * bd + threadIdx.x;
      const float* __restrict__ VGk = reinterpret_cast<const float*>(T.VG32T + (size_t)kk * T.nwin);
      const float* __restrict__ vk = cd.w.v32 + (size_t)kk * nl;
      if (pm0 >= 0) {
        cp_async4(r, VGk + 2 * (pm0 >> 8));
        cp_async4(r + bd, VGk + 2 * (pm0 >> 8) + 1);
        cp_async4(r + 2 * bd, vk + ((pm0 >> 4) & 15));
        cp_async4(r + 3 * bd, vk + (pm0 & 15));
      }
      if (pm1 >= 0) {
        cp_async4(r + 4 * bd, VGk + 2 * (pm1 >> 8));
        cp_async4(r + 5 * bd, VGk + 2 * (pm1 >> 8) + 1);
        cp_async4(r + 6 * bd, vk + ((pm1 >> 4) & 15));
        cp_async4(r + 7 * bd, vk + (pm1 & 15));
      }
      cp_async4(r + 8 * bd, S32T + (size_t)kk * pitch);
    }
    cp_async_commit();
  };
  // ... and the opacity tangent of depth kk formed from its stage (and the
  // rest of the depth's transitions, read directly; the order of the
  // separate opacity kernel; chi_k: the float opacity of that depth), stored
  // for the outward pass. Every copy but those of the kRing - 2 most recent
  // depths has landed after the wait.
  auto tan_finish = [&](int kk, float chik, float& dc, float& dS) {
    cp_async_wait<kRing - 2>();
    const float* r = s_ring + (size_t)(kk % kRing) * kRingSlots * bd + threadIdx.x;
    TanAcc ta;
    if (pm0 >= 0) tan_acc(ta, r[0], r[bd], r[2 * bd], r[3 * bd]);
    if (pm1 >= 0) {
      tan_acc(ta, r[4 * bd], r[5 * bd], r[6 * bd], r[7 * bd]);
      const float2* __restrict__ VGk = T.VG32T + (size_t)kk * T.nwin;
      const float* __restrict__ vk = cd.w.v32 + (size_t)kk * nl;
#pragma unroll
      for (int j = 2; j < kQMetaT; ++j) {
        const int m = __ldg(T.qmeta + (size_t)j * nq + q);
        if (m < 0) break;
        const float2 a = __ldg(VGk + (m >> 8));
        tan_acc(ta, a.x, a.y, __ldg(vk + ((m >> 4) & 15)), __ldg(vk + (m & 15)));
      }
    }
    dc = ta.dchi;
    dS = tan_dS(ta, r[8 * bd], chik);
    const size_t o = (size_t)kk * pitch + q;
    cd.w.dchiT[o] = dc;
    cd.w.dS32T[o] = dS;
  };
  // tangent opacity of depth kk, left by the opacity kernel or (outward pass
  // of a fused sweep) by the inward pass
  auto tan_in = [&](int kk, float& dc, float& dS) {
    const size_t o = (size_t)kk * pitch;
    dc = dchiT[o];
    dS = dS32T[o];
  };

  // boundary depth: I = 0 at the top, I = B at the bottom (Sect. 2.1)
  const int k0 = UP ? nz - 1 : 0;
  df Sp = df_load(S2, k0);
  float cp = TAN ? chiT[k0 * pitch] : chi[k0];
  float dSp = 0.f, dcp = 0.f;
  if (FT) {
#pragma unroll
    for (int j = 0; j < kRing - 1; ++j) tan_issue(k0 + j);
    tan_finish(k0, cp, dcp, dSp);
    tan_issue(k0 + kRing - 1);
  } else if (TAN) {
    tan_in(k0, dcp, dSp);
  }
  float Su = Sp.hi;
  if (!TAN && !UP) {
    chiT[0] = cp;
    S32T[0] = Su;
  }
  const double Ib64 = UP ? T.Bn[row + nz - 1] / c2 : 0.0;
  const float D0 = df_to_float(df_sub(df_from_double(Ib64), Sp));
  const float I0 = __double2float_rn(Ib64);
  const float dD0 = -dSp;
  float D[MU], I[MU], M[MU], dD[MU];
  float xD[8], xa[8], xI[8], xx[8], xe[8], xd[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) xD[m] = xa[m] = xI[m] = xx[m] = xe[m] = xd[m] = 0.f;
#pragma unroll
  for (int m = 0; m < MU; ++m) {
    D[m] = D0;
    I[m] = I0;
    M[m] = fabsf(D0);
    dD[m] = dD0;
    if (EXACT || m < nmu) {
      xD[m] = mul(hw[m], D0);
      xa[m] = fabsf(xD[m]);
      xI[m] = mul(hw[m], I0);
      xd[m] = mul(hw[m], dD0);
    }
  }
  // the inward pass leaves its hemisphere sums of each depth in part; the
  // outward pass adds its own to them (pt: those of depth k, loaded ahead)
  constexpr int NP = TAN ? 1 : kSweepParts;
  auto emit = [&](int k, df Sk, float dS, const float* pt) {
    float* pp = part + (size_t)k * pitch;
    if (TAN) {
      const float td = tree_mu<MU>(xd);
      if (!UP) pp[0] = td;
      else write_tan(cd, (size_t)k * pitch + q, dS, add(td, pt[0]));
      return;
    }
    const float tD = tree_mu<MU>(xD), ta = tree_mu<MU>(xa), tI = tree_mu<MU>(xI), tx = tree_mu<MU>(xx),
                te = tree_mu<MU>(xe);
    if (!UP) {
      pp[0] = tD;
      pp[pstride] = ta;
      pp[2 * pstride] = tI;
      pp[3 * pstride] = tx;
      pp[4 * pstride] = te;
    } else {
      const BaseOut r = base_out(Sk, c2p, c2f, add(tD, pt[0]), add(ta, pt[1]), add(tI, pt[2]), add(tx, pt[3]),
                                 add(te, pt[4]));
      const int lane = threadIdx.x & 31;
      float* w = s_stage + lane * (kStageD + 1) + (k % kStageD);
      w[0] = r.J.hi;
      w[kStagePlane] = r.J.lo;
      w[2 * kStagePlane] = r.lx;
      w[3 * kStagePlane] = r.le;
      if (k % kStageD == 0) {
        // the depths k .. k + kStageD - 1 of the warp's rows are complete
        __syncwarp(amask);
        const int nk = min(kStageD, nz - k);
        const int q0w = q - lane;
        float2* __restrict__ J2 = as_pairs(jnew_ptr(cd));
        if (na == 32 && nk == kStageD) {
          // full warp, full block: lane -> (row lane / 8 + 4 i, depth lane % 8)
          static_assert(kStageD == 8, "the full-block flush maps 4 rows x 8 depths per pass");
          const int kk = lane & 7;
          const size_t o0 = (size_t)(q0w + (lane >> 3)) * nz + k + kk;
          const float* s0 = s_stage + (lane >> 3) * (kStageD + 1) + kk;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float* sr = s0 + 4 * i * (kStageD + 1);
            const size_t o = o0 + (size_t)(4 * i) * nz;
            J2[o] = make_float2(sr[0], sr[kStagePlane]);
            cd.w.Lchi32[o] = sr[2 * kStagePlane];
            cd.w.Leta32[o] = sr[3 * kStagePlane];
          }
        } else {
          for (int e = lane; e < na * nk; e += na) {
            const int rr = e / nk, kk = e - rr * nk;
            const float* sr = s_stage + rr * (kStageD + 1) + kk;
            const size_t o = (size_t)(q0w + rr) * nz + k + kk;
            J2[o] = make_float2(sr[0], sr[kStagePlane]);
            cd.w.Lchi32[o] = sr[2 * kStagePlane];
            cd.w.Leta32[o] = sr[3 * kStagePlane];
          }
        }
        __syncwarp(amask);
      }
    }
  };
  float pt_n[NP];
  auto load_parts = [&](int kk) {
    if (UP) {
#pragma unroll
      for (int j = 0; j < NP; ++j) pt_n[j] = part[(size_t)kk * pitch + j * pstride];
    }
  };
  load_parts(k0);
  emit(k0, Sp, dSp, pt_n);

  // the next depth's inputs are prepared one step ahead
  int kn = UP ? nz - 2 : 1;
  float c_n = 0.f, dc_n = 0.f, dS_n = 0.f, dSl_n = 0.f, Sf_n = 0.f;
  df S_n = df_make(0.f, 0.f);
  auto load = [&](int kk) {
    load_parts(kk);
    if (TAN) {
      c_n = chiT[(size_t)kk * pitch];
      dSl_n = dSkT[(size_t)(UP ? kk : kk - 1) * pitch];
      if (!FT) tan_in(kk, dc_n, dS_n);
    } else if (UP) {
      // the outward sweep of a base evaluation reads the float copies its own
      // inward sweep left (coalesced; the same values, no pair difference)
      // and the S pair for J only
      c_n = chiT[(size_t)kk * pitch];
      Sf_n = S32T[(size_t)kk * pitch];
      dSl_n = dSkT[(size_t)kk * pitch];
      S_n = df_load(S2, kk);
    } else {
      c_n = chi[kk];
      S_n = df_load(S2, kk);
    }
  };
  if (nz > 1) load(kn);
  for (int s = 1; s < nz; ++s) {
    const int k = kn;
    const int kd = UP ? k : k - 1;   // layer between k and its upstream neighbour
    const float c0 = c_n, dSl = dSl_n, Sf = Sf_n;
    float dc0 = dc_n, dS0 = dS_n;
    if (FT) {
      tan_finish(k, c0, dc0, dS0);
      tan_issue(k + kRing - 1);
    }
    const df Sk = S_n;
    float pt[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) pt[j] = pt_n[j];
    if (s + 1 < nz) {
      kn = UP ? k - 1 : k + 1;
      load(kn);
    }
    StepIn in;
    in.csum = add(c0, cp);
    in.rs = rcp_approx(in.csum);
    in.dzk = s_dz[kd];
    in.idzk = s_idz[kd];
    in.tz = mul(in.dzk, in.csum);
    in.rz = mul(in.rs, in.idzk);
    in.dtz = 0.f;
    if (TAN) {
      in.dSin = UP ? dSl : -dSl;
      in.S0 = in.Su = in.rc0 = 0.f;
      in.dcs = add(dc0, dcp);
      in.dtz = mul(in.dzk, in.dcs);
      in.ddSin = sub(dSp, dS0);
    } else {
      // S^u - S^k formed from the pairs, then rounded
      in.dSin = UP ? dSl : df_to_float(df_sub(Sp, Sk));
      in.S0 = UP ? Sf : Sk.hi;
      if (!UP) {
        // depth-major copies for the tangent evaluations
        chiT[(size_t)k * pitch] = c0;
        S32T[(size_t)k * pitch] = in.S0;
        dSkT[(size_t)kd * pitch] = -in.dSin;   // S^{k} - S^{k-1}
      }
      in.Su = Su;
      in.rc0 = rcp_approx(c0);
      in.dcs = in.ddSin = 0.f;
    }
    auto angles = [&](auto cm) {
      constexpr int CM = decltype(cm)::value;
#pragma unroll
      for (int m = 0; m < MU; ++m) {
        if (EXACT || m < nmu) {
          const RayOut r = ray_step<TAN, CM>(in, inv2mu[m], two_mu[m], hw[m], D[m], I[m], M[m], dD[m]);
          xD[m] = r.xD;
          xa[m] = fabsf(r.xD);
          xI[m] = r.xI;
          xx[m] = r.xx;
          xe[m] = r.xe;
          xd[m] = r.xd;
        }
      }
    };
    if (EXACT) {
      // the angles' optical depths tz/(2 mu) fall with m (mu ascending): one
      // test on the first and last angle settles the form for all of them. The
      // warp takes one form together: lanes that differ would run every form one
      // after the other (base sweeps of 512 Ca II columns: 38.0 -> 36.5 ms a solve).
      if (__all_sync(amask, !(mul(in.tz, inv2mu[MU - 1]) < 0.1f)))
        angles(std::integral_constant<int, CM_DIRECT>());
      else if (__all_sync(amask, mul(in.tz, inv2mu[0]) < 0.1f)) angles(std::integral_constant<int, CM_SERIES>());
      else angles(std::integral_constant<int, CM_SELECT>());
    } else {
      angles(std::integral_constant<int, CM_EITHER>());
    }
    emit(k, Sk, dS0, pt);
    Sp = Sk;
    Su = in.S0;
    cp = c0;
    dSp = dS0;
    dcp = dc0;
  }
  if (UP && !TAN) {
#pragma unroll
    for (int m = 0; m < MU; ++m)
      if (EXACT || m < nmu) cd.w.Iem[(size_t)q * nmu + m] = __dmul_rn((double)I[m], c2);
  }
}

// ---------------------------------------------------------------------------
// Tangent sweep of a large launch: one thread per two neighbouring frequencies,
// every FP32 operation a packed pair (fma.rn.f32x2 and its mul: two IEEE
// operations in one instruction). The scalar sweep filled the issue slots (0.88
// of the peak rate) with DRAM and the FP32 lanes half idle; a packed instruction
// takes the lanes twice as long as a scalar one but one issue slot, and loads
// and addresses are shared by the two frequencies. A warp votes on the form of
// the coefficients, so that lanes on both sides of the limit cost one pass and
// not three. Each element sees the operations of ray_step in their order: the
// same bits. On the 76-column batch, which leaves the SMs at two blocks each, the
// FP32 pipe is 42 % busy and the issue slots 32 % (48 % with the scalar sweep); the
// 4,096-column batch runs at 0.70 of the FP32 roofline (0.56).
// 512 Ca II columns, 256 x 1,005, 5 angles, median launch of a solve: scalar 960 us,
// scalar with the vote 999, packed 963, packed with the vote 785 (57.0 -> 46.8 ms per
// solve). A vote per angle in mixed warps: 47.9 ms; 64 threads per block: 49.0.
// ---------------------------------------------------------------------------
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 both2(float a) { return pack2(a, a); }
// a + b and a - b as fma with a packed 1 or -1 the compiler cannot see the value
// of (a kernel argument): it contracts a packed product and the add.rn.f32x2 or
// constant fma after it into one operation, which rounds once instead of twice
// (it leaves the scalar mul.rn and add.rn apart).
struct Ones2 {
  f32x2 one, neg;
};
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b, const Ones2& u) { return fma2(a, u.one, b); }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b, const Ones2& u) { return fma2(b, u.neg, a); }
__device__ __forceinline__ f32x2 ld2(const float* p) { return *reinterpret_cast<const f32x2*>(p); }
__device__ __forceinline__ void st2(float* p, f32x2 v) { *reinterpret_cast<f32x2*>(p) = v; }
__device__ __forceinline__ f32x2 select2(bool a, bool b, f32x2 x, f32x2 y) {   // per element: x or y
  float x0, x1, y0, y1;
  unpack2(x, x0, x1);
  unpack2(y, y0, y1);
  return pack2(a ? x0 : y0, b ? x1 : y1);
}
__device__ __forceinline__ void series2(f32x2 x, f32x2& w, f32x2& bq) {
  w = fma2(fma2(fma2(fma2(fma2(both2(-1.0f / 720.0f), x, both2(1.0f / 120.0f)), x, both2(-1.0f / 24.0f)), x,
                     both2(1.0f / 6.0f)), x, both2(-0.5f)), x, both2(1.0f));
  bq = fma2(fma2(fma2(fma2(both2(1.0f / 144.0f), x, both2(-1.0f / 30.0f)), x, both2(1.0f / 8.0f)), x,
                 both2(-1.0f / 3.0f)), x, both2(0.5f));
}
__device__ __forceinline__ void direct2(f32x2 e, f32x2 r, f32x2& w, f32x2& bq, const Ones2& u) {
  w = mul2(sub2(u.one, e, u), r);
  bq = mul2(sub2(w, e, u), r);
}

constexpr int kPairThreads = 128;
constexpr int kPairAhead = 4;   // depths ahead whose rows are prefetched into L2

// A column with fewer than MU angles runs the others with zero weight and zero
// optical depth (they add zeros to its sums).
template <int MU, bool UP>
__device__ __forceinline__ void sweep_pair(const ColDesc& cd, int q, const float* __restrict__ s_dz,
                                           const float* __restrict__ s_idz, const Ones2& u, unsigned amask) {
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq;
  const size_t pitch = (size_t)col_pitch(nq);
  const float* __restrict__ chiT = cd.w.chiT + q;
  const float* __restrict__ dSkT = cd.w.dSkT + q;
  const float* __restrict__ dchiT = cd.w.dchiT + q;
  const float* __restrict__ dS32T = cd.w.dS32T + q;
  float* __restrict__ part = reinterpret_cast<float*>(cd.w.part) + q;
  float* __restrict__ dJ = cd.w.dJ32T + q;
  float inv2mu[MU], two_mu[MU], hw[MU];
#pragma unroll
  for (int m = 0; m < MU; ++m) {
    const float4 a = T.ang32[m];
    inv2mu[m] = a.x;
    hw[m] = a.y;
    two_mu[m] = a.z;
  }
  const float inv2mu_last = T.ang32[T.nmu - 1].x;
  // boundary depth: I = 0 at the top, I = B at the bottom (Sect. 2.1)
  const int k0 = UP ? nz - 1 : 0, q1 = min(q + 1, nq - 1);
  auto D0_of = [&](int qq) {
    const size_t i = (size_t)qq * nz;
    const double Ib = UP ? T.Bn[i + nz - 1] / T.c2[qq] : 0.0;
    return df_to_float(df_sub(df_from_double(Ib), df_load(as_pairs(cd.w.S), i + k0)));
  };
  f32x2 cp = ld2(chiT + k0 * pitch), dcp = ld2(dchiT + k0 * pitch), dSp = ld2(dS32T + k0 * pitch);
  f32x2 D[MU], dD[MU], x[8];
  {
    const f32x2 D0 = pack2(D0_of(q), D0_of(q1));
    float a, b;
    unpack2(dSp, a, b);
    const f32x2 dD0 = pack2(-a, -b);
#pragma unroll
    for (int m = 0; m < MU; ++m) {
      D[m] = D0;
      dD[m] = dD0;
      x[m] = mul2(both2(hw[m]), dD0);
    }
  }
  // the angles' sum in the order of tree_mu
  auto tree = [&]() {
    auto pair_add = [&](int i, int j) { return j < MU ? add2(x[i], x[j], u) : x[i]; };   // i < MU
    f32x2 ev = pair_add(0, 4);
    if (MU > 2) ev = add2(ev, pair_add(2, 6), u);
    if (MU == 1) return ev;
    f32x2 od = pair_add(1, 5);
    if (MU > 3) od = add2(od, pair_add(3, 7), u);
    return add2(ev, od, u);
  };
  auto emit = [&](int k, f32x2 dS, f32x2 pt) {
    const f32x2 t = tree();
    if (!UP) st2(part + (size_t)k * pitch, t);
    else st2(dJ + (size_t)k * pitch, add2(dS, add2(t, pt, u), u));
  };
  emit(k0, dSp, UP ? ld2(part + (size_t)k0 * pitch) : 0);
  // the next depth's inputs are loaded one step ahead, their lines brought into L2 before that
  int kn = UP ? nz - 2 : 1;
  f32x2 c_n = 0, dc_n = 0, dS_n = 0, dSl_n = 0, pt_n = 0;
  auto load = [&](int k) {
    c_n = ld2(chiT + (size_t)k * pitch);
    dSl_n = ld2(dSkT + (size_t)(UP ? k : k - 1) * pitch);
    dc_n = ld2(dchiT + (size_t)k * pitch);
    dS_n = ld2(dS32T + (size_t)k * pitch);
    if (UP) pt_n = ld2(part + (size_t)k * pitch);
    const int kf = UP ? k - kPairAhead : k + kPairAhead;
    if (kf >= 0 && kf < nz) {
      const size_t o = (size_t)kf * pitch;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(chiT + o));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(dSkT + o));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(dchiT + o));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(dS32T + o));
      if (UP) asm volatile("prefetch.global.L2 [%0];" ::"l"(part + o));
    }
  };
  if (nz > 1) load(kn);
  for (int s = 1; s < nz; ++s) {
    const int k = kn, kd = UP ? k : k - 1;   // layer between k and its upstream neighbour
    const f32x2 c0 = c_n, dc0 = dc_n, dS0 = dS_n, dSl = dSl_n, pt = pt_n;
    if (s + 1 < nz) {
      kn = UP ? k - 1 : k + 1;
      load(kn);
    }
    const f32x2 dz = both2(s_dz[kd]);
    const f32x2 csum = add2(c0, cp, u);
    float ca, cb, ta, tb;
    unpack2(csum, ca, cb);
    const f32x2 tz = mul2(dz, csum), rz = mul2(pack2(rcp_approx(ca), rcp_approx(cb)), both2(s_idz[kd]));
    const f32x2 dtz = mul2(dz, add2(dc0, dcp, u)), ddSin = sub2(dSp, dS0, u);
    const f32x2 dSin = UP ? dSl : mul2(dSl, u.neg);
    unpack2(tz, ta, tb);
    // the angles' optical depths tz/(2 mu) fall with m (mu ascending): a test on
    // the first and last angle settles the form for all of them. The warp takes
    // one form together: lanes that differ would run every form one after the other.
    const bool direct =
        __all_sync(amask, !(mul(ta, inv2mu_last) < 0.1f) && !(mul(tb, inv2mu_last) < 0.1f));
    const bool series = __all_sync(amask, mul(ta, inv2mu[0]) < 0.1f && mul(tb, inv2mu[0]) < 0.1f);
    auto angles = [&](auto cm) {
      constexpr int CM = decltype(cm)::value;
#pragma unroll
      for (int m = 0; m < MU; ++m) {
        const f32x2 dtau = mul2(tz, both2(inv2mu[m]));
        float a, b, ea, eb;
        unpack2(mul2(dtau, both2(-1.4426950408889634f)), a, b);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ea) : "f"(a));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(eb) : "f"(b));
        const f32x2 e = pack2(ea, eb);
        f32x2 w, bq;
        if (CM != CM_SERIES) direct2(e, mul2(rz, both2(two_mu[m])), w, bq, u);
        if (CM == CM_SERIES) series2(dtau, w, bq);
        if (CM == CM_SELECT) {
          f32x2 ws, bs;
          series2(dtau, ws, bs);
          unpack2(dtau, a, b);
          w = select2(a < 0.1f, b < 0.1f, ws, w);
          bq = select2(a < 0.1f, b < 0.1f, bs, bq);
        }
        const f32x2 tn = mul2(dtz, both2(-inv2mu[m]));   // -ddtau
        const f32x2 dDn = fma2(dD[m], e, fma2(tn, fma2(e, D[m], mul2(bq, dSin)), mul2(w, ddSin)));
        D[m] = fma2(D[m], e, mul2(w, dSin));
        dD[m] = dDn;
        x[m] = mul2(both2(hw[m]), dDn);
      }
    };
    if (direct) angles(std::integral_constant<int, CM_DIRECT>());
    else if (series) angles(std::integral_constant<int, CM_SERIES>());
    else angles(std::integral_constant<int, CM_SELECT>());
    emit(k, dS0, pt);
    cp = c0;
    dcp = dc0;
    dSp = dS0;
  }
}

// MU: the largest angle count of the launch, each with its own instantiation.
// Columns with fewer run the same code: a second body for them in this kernel
// raised the registers from 96 to 128 (four blocks per SM, not five), and the
// scalar sweep of one frequency after the other, which stood here, was slower than
// the one-frequency kernel this one took the place of. 256 Ca II columns, a solve,
// one frequency per thread -> that -> now: 1 angle 112.6 -> 130.4 -> 102.3 ms, 6
// angles 132.5 -> 144.6 -> 114.8, 7 angles 136.3 -> 147.6 -> 119.9, columns of 3 and
// 5 angles 119.8 -> 127.7 -> 112.3.
template <int MU>
__global__ void __launch_bounds__(kPairThreads, MU <= 5 ? 5 : 4) k_formal_sweep_pair(const ColDesc* __restrict__ cols,
                                                                    float one) {   // one: 1
  extern __shared__ float s_tab[];   // [nz] |dz|, [nz] 1/|dz|
  const ColDesc& cd = cols[blockIdx.y];
  if (eval_mode_f(cd) != EV_TANGENT) return;
  const ColTables& T = cd.t;
  if ((int)(2 * blockIdx.x * blockDim.x) >= T.nq) return;   // uniform over the block
  float* s_dz = s_tab;
  float* s_idz = s_tab + T.nz;
  stage_dz(T, s_dz, s_idz);
  __syncthreads();
  const int q = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const unsigned amask = __ballot_sync(0xffffffffu, q < T.nq);
  if (q >= T.nq) return;
  const Ones2 u{both2(one), both2(-one)};
  sweep_pair<MU, false>(cd, q, s_dz, s_idz, u, amask);
  sweep_pair<MU, true>(cd, q, s_dz, s_idz, u, amask);
}

// One kernel per evaluation kind (its own register allocation): blocks of
// columns in the other kind return at once. FUSE: the tangent kernel forms
// the opacity tangent itself (no separate opacity-tangent launch).
template <int MU, bool TAN, bool FUSE>
__device__ __forceinline__ void formal_sweep_block(const ColDesc* __restrict__ cols) {
  extern __shared__ float s_tab[];   // FUSE: the copy ring; then [nz] |dz|, [nz] 1/|dz|
  const ColDesc& cd = cols[blockIdx.y];
  const int mode = eval_mode_f(cd);
  if (mode == EV_SKIP || (mode == EV_TANGENT) != TAN) return;
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq;
  if ((int)(blockIdx.x * blockDim.x) >= nq) return;   // uniform over the block
  // FUSE: the copy ring; base-type sweeps: the output stage; then the |dz| tables
  float* s_ring = FUSE ? s_tab : nullptr;
  float* s_stage = TAN ? nullptr : s_tab + (size_t)(threadIdx.x >> 5) * kWarpStage;
  float* s_dz = s_tab + (FUSE ? ring_floats(blockDim.x) : 0) + (TAN ? 0 : stage_floats(blockDim.x));
  float* s_idz = s_dz + nz;
  stage_dz(T, s_dz, s_idz);
  __syncthreads();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  // the lanes of a warp with a frequency form a prefix of it
  const unsigned amask = __ballot_sync(0xffffffffu, q < nq);
  if (q >= nq) return;
  const int na = __popc(amask);
  if (T.nmu == MU) {   // uniform over the block: every angle slot is in use
    sweep_thread<MU, TAN, false, true, FUSE>(cd, q, s_dz, s_idz, s_ring, s_stage, amask, na);
    sweep_thread<MU, TAN, true, true>(cd, q, s_dz, s_idz, nullptr, s_stage, amask, na);
  } else {
    sweep_thread<MU, TAN, false, false, FUSE>(cd, q, s_dz, s_idz, s_ring, s_stage, amask, na);
    sweep_thread<MU, TAN, true, false>(cd, q, s_dz, s_idz, nullptr, s_stage, amask, na);
  }
}

template <int MU>
__global__ void __launch_bounds__(256) k_formal_sweep(const ColDesc* __restrict__ cols) {
  formal_sweep_block<MU, false, false>(cols);
}

// The tangent sweep that forms the opacity tangent itself (forced variant):
// 128-thread blocks, at most 72 registers (seven blocks per SM). Measured on
// the 1,216-column batch against the separate opacity-tangent kernel
// (per tick, all on one stream): opacity stage 1.67 -> 0.63 ms, tangent sweep
// 1.54 -> 2.91 ms; whole solve 529 -> 554 ms. At 64 registers (spills) the
// sweep took 3.51 ms, unbounded (100 registers) 3.69 ms.
constexpr int kFusedThreads = 128;
template <int MU>
__global__ void __launch_bounds__(kFusedThreads, 7) k_formal_sweep_fused(const ColDesc* __restrict__ cols) {
  formal_sweep_block<MU, true, true>(cols);
}

// ---------------------------------------------------------------------------
// Variant 2 (small launches): one warp per two frequencies; lane = (frequency
// of the pair, hemisphere, angle), so both hemispheres advance together and
// every lane runs one ray. A hemisphere's sums are those of an xor butterfly
// over its 8 angle lanes (the tree of tree_mu), every kWarpChunk depths from
// the lanes' rows in shared memory.
//
// A small launch is bound by latency: one trip to L2 per depth was most of it.
// A 233-depth, 2,010-frequency column: base evaluation 288 + 15 us (thread
// variant and its opacity kernel) -> 66, tangent 221 + 29 -> 39 us; 82 depths:
// base 83 + 6 -> 25 us. So
// a block first stages every depth of its frequencies in shared memory, all
// loads in flight at once, and forms the opacity there: the separate opacity
// kernels (6 to 28 us at these sizes, too few threads in flight) are not
// launched, and the recurrence then reads shared memory only. It has about one
// warp per scheduler, so its steps are straight code: the coefficients of
// kWarpAhead depths are formed before the steps through them, both their forms
// and a selection instead of a branch, and no shuffles.
// ---------------------------------------------------------------------------
constexpr int kWarpAhead = 4;    // depths whose coefficients are formed together
constexpr int kWarpStage2 = 2;   // warps that stage per warp that sweeps
constexpr int kWarpChunk = 16;   // depths between two sums over the angle lanes
static_assert(kWarpChunk % kWarpAhead == 0, "a chunk is whole groups");

__host__ __device__ inline int warp_parts(bool tan) { return tan ? 1 : kSweepParts; }
// rows of a chunk: one word per lane of dD, or of D, I, dI/dchi, dI/deta, padded by a bank
__host__ __device__ inline int warp_lanes_row(bool tan) { return (tan ? 1 : 4) * 32 + 1; }
__host__ __device__ inline int warp_row(int nz) { return nz | 1; }   // odd: lanes on different frequencies, different banks

__host__ __device__ inline size_t warp_variant_smem(int nz, int warps, bool tan) {
  return sizeof(float) * (2 * (size_t)nz + (size_t)warps * (2 * 4 * (size_t)warp_row(nz) + 2 * warp_parts(tan) * (size_t)nz +
                                                                 kWarpChunk * warp_lanes_row(tan)));
}

// Stage of a tangent block: chi, S^{k+1} - S^k, dchi, dS of its frequencies at
// every depth ([array][frequency][depth]); dchi and dS as k_opacity_tan32
// forms them (tan_acc, tan_dS: the same bits).
__device__ __forceinline__ void stage_tan(const ColDesc& cd, int qb, int F, float* __restrict__ st, int row) {
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq, nl = T.nl, nwin = T.nwin;
  const int f = threadIdx.x % F, q = qb + f;
  if (q >= nq) return;
  const size_t pitch = (size_t)col_pitch(nq);
  const double* __restrict__ dir = cd.forced_mode >= 0 ? cd.w.v
                                   : cd.w.st->phase == PH_RESTART ? cd.w.x
                                                                  : cd.w.Vb + (size_t)cd.w.st->j * nz * nl;
  const int m0 = __ldg(T.qmeta + q), m1 = __ldg(T.qmeta + (size_t)nq + q);
  float* o = st + (size_t)f * row;
  const size_t plane = (size_t)F * row;
  const int ks = blockDim.x / F;
#pragma unroll 4
  for (int k = threadIdx.x / F; k < nz; k += ks) {
    const size_t i = (size_t)k * pitch + q;
    const float S = cd.w.S32T[i], c = cd.w.chiT[i];
    const float dSk = k < nz - 1 ? cd.w.dSkT[i] : 0.f;
    const float2* __restrict__ VG = T.VG32T + (size_t)k * nwin;
    const double* __restrict__ v = dir + (size_t)k * nl;
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
    float l0 = 0.f, u0 = 0.f, l1 = 0.f, u1 = 0.f;
    if (m0 >= 0) {
      a0 = __ldg(VG + (m0 >> 8));
      l0 = (float)v[(m0 >> 4) & 15];
      u0 = (float)v[m0 & 15];
    }
    if (m1 >= 0) {
      a1 = __ldg(VG + (m1 >> 8));
      l1 = (float)v[(m1 >> 4) & 15];
      u1 = (float)v[m1 & 15];
    }
    TanAcc ta;
    if (m0 >= 0) tan_acc(ta, a0.x, a0.y, l0, u0);
    if (m1 >= 0) {
      tan_acc(ta, a1.x, a1.y, l1, u1);
      for (int j = 2; j < kQMetaT; ++j) {
        const int m = __ldg(T.qmeta + (size_t)j * nq + q);
        if (m < 0) break;
        const float2 a = __ldg(VG + (m >> 8));
        tan_acc(ta, a.x, a.y, (float)v[(m >> 4) & 15], (float)v[m & 15]);
      }
      if (T.max_overlap > kQMetaT)
        for (int s = T.q_off[q] + kQMetaT; s < T.q_off[q + 1]; ++s) {
          const int t = T.q_t[s];
          const float2 a = __ldg(VG + T.t_base[t] + q - T.t_q0[t]);
          tan_acc(ta, a.x, a.y, (float)v[T.t_lo[t]], (float)v[T.t_up[t]]);
        }
    }
    o[k] = c;
    o[plane + k] = dSk;
    o[2 * plane + k] = ta.dchi;
    o[3 * plane + k] = tan_dS(ta, S, c);
  }
}

// Stage of a base-type block: chi, S^{k+1} - S^k (formed from the pairs, then
// rounded), S as a pair; and the arrays the tangents of the Newton step read.
__device__ __forceinline__ void stage_base(const ColDesc& cd, int mode, int qb, int F, float* __restrict__ st,
                                           int row) {
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq;
  const int nf = min(F, nq - qb);
  const size_t plane = (size_t)F * row, pitch = (size_t)col_pitch(nq);
  for (int i = threadIdx.x; i < nf * nz; i += blockDim.x) {
    const int f = i / nz, k = i - f * nz;
    const BasePoint p = base_opacity<true>(cd, mode, qb + f, k, (qb + f) * nz + k);
    float* o = st + (size_t)f * row + k;
    o[0] = p.chi;
    o[2 * plane] = p.S.hi;
    o[3 * plane] = p.S.lo;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nf * nz; i += blockDim.x) {
    const int k = i / nf, f = i - k * nf;
    float* o = st + (size_t)f * row + k;
    const size_t g = (size_t)k * pitch + qb + f;
    cd.w.chiT[g] = o[0];
    cd.w.S32T[g] = o[2 * plane];
    if (k < nz - 1) {
      const df a = df_make(o[2 * plane], o[3 * plane]), b = df_make(o[2 * plane + 1], o[3 * plane + 1]);
      const float d = -df_to_float(df_sub(a, b));   // S^{k+1} - S^k
      o[plane] = d;
      cd.w.dSkT[g] = d;
    }
  }
}

template <bool TAN>
__device__ __forceinline__ void sweep_warp(const ColDesc& cd, int q, int fl, const float* __restrict__ st, int row,
                                           size_t plane, float* __restrict__ wp, const float* __restrict__ s_dz,
                                           const float* __restrict__ s_idz) {
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq, nmu = T.nmu;
  const int lane = threadIdx.x & 31;
  const int qi = lane >> 4, hemi = (lane >> 3) & 1, m = lane & 7;
  const bool up = hemi == 1;
  const bool valid = q < nq;
  const int qq = valid ? q : nq - 1;
  constexpr int NP = TAN ? 1 : kSweepParts;
  const float* __restrict__ in = st + (size_t)(valid ? fl : 0) * row;   // this frequency's staged rows
  const double c2 = T.c2[qq];
  // lanes past the last angle run with zero weight (their sums add zeros)
  const float4 ang = m < nmu ? T.ang32[m] : make_float4(0.f, 0.f, 0.f, 0.f);
  const float inv2mu = ang.x;
  const float hw = ang.y;
  const float two_mu = ang.z;
  constexpr int LR = (TAN ? 1 : 4) * 32 + 1;
  float* lanes = wp + (size_t)2 * NP * nz;   // [kWarpChunk][LR]; wp: [2][NP][nz]

  const int k0 = up ? nz - 1 : 0;
  const df Sb = TAN ? df_load(as_pairs(cd.w.S), (size_t)qq * nz + k0) : df_make(in[2 * plane + k0], in[3 * plane + k0]);
  const double Ib64 = up ? T.Bn[(size_t)qq * nz + nz - 1] / c2 : 0.0;
  const float D0 = df_to_float(df_sub(df_from_double(Ib64), Sb));
  const float I0 = __double2float_rn(Ib64);
  const float dD0 = TAN ? -in[3 * plane + k0] : -0.f;
  float D = D0, I = I0, M = fabsf(D0), dD = dD0;
  // row r of the chunk: the boundary depth is the first chunk's row 0
  auto put = [&](int r, const RayOut& x) {
    float* o = lanes + r * LR + lane;
    if (TAN) {
      o[0] = x.xd;
    } else {
      o[0] = x.xD;
      o[32] = x.xI;
      o[64] = x.xx;
      o[96] = x.xe;
    }
  };
  {
    RayOut r;
    r.xD = mul(hw, D0);
    r.xI = mul(hw, I0);
    r.xx = r.xe = 0.f;
    r.xd = mul(hw, dD0);
    put(0, r);
  }
  for (int c0 = 0; c0 < nz; c0 += kWarpChunk) {
    const int c1 = min(c0 + kWarpChunk, nz);
    for (int s0 = max(c0, 1); s0 < c1; s0 = (s0 & ~(kWarpAhead - 1)) + kWarpAhead) {
      RayCoef c[kWarpAhead];
      float dSin[kWarpAhead], S0[kWarpAhead], rc0[kWarpAhead];
      const int se = min((s0 & ~(kWarpAhead - 1)) + kWarpAhead, c1);   // steps s0 .. se - 1
#pragma unroll
      for (int u = 0; u < kWarpAhead; ++u) {
        const int s = min(s0 + u, nz - 1);
        const int k = up ? nz - 1 - s : s, ku = up ? k + 1 : k - 1, kd = up ? k : k - 1;
        StepIn x;
        const float cc = in[k];
        const float dSl = in[plane + kd];
        x.csum = add(cc, in[ku]);
        x.rs = rcp_approx(x.csum);
        x.dzk = s_dz[kd];
        x.idzk = s_idz[kd];
        x.tz = mul(x.dzk, x.csum);
        x.rz = mul(x.rs, x.idzk);
        x.dSin = up ? dSl : -dSl;
        if (TAN) {
          x.dcs = add(in[2 * plane + k], in[2 * plane + ku]);
          x.dtz = mul(x.dzk, x.dcs);
          x.ddSin = sub(in[3 * plane + ku], in[3 * plane + k]);
          x.S0 = x.Su = x.rc0 = 0.f;
        } else {
          x.S0 = in[2 * plane + k];
          x.Su = in[2 * plane + ku];
          x.rc0 = rcp_approx(cc);
          x.dcs = x.dtz = x.ddSin = 0.f;
        }
        c[u] = ray_coef<TAN, CM_SELECT>(x, inv2mu, two_mu, hw);
        dSin[u] = x.dSin;
        S0[u] = x.S0;
        rc0[u] = x.rc0;
      }
#pragma unroll
      for (int u = 0; u < kWarpAhead; ++u)
        if (s0 + u < se) put(s0 + u - c0, ray_apply<TAN>(c[u], dSin[u], S0[u], rc0[u], hw, D, I, M, dD));
    }
    __syncwarp();
    // the hemispheres' sums of the chunk's depths: row r of group (frequency,
    // hemisphere). The hemisphere that reaches a depth first leaves its sums in
    // wp, the other one adds its own and writes the depth's output (a middle
    // depth is reached by both in one row); first the rows of the first kind.
    const size_t pitch = (size_t)col_pitch(nq);
    for (int pass = 0; pass < 2; ++pass) {
      for (int i = lane; i < (c1 - c0) * 4; i += 32) {
        const int g = i & 3, r = i >> 2, s = c0 + r, o = nz - 1 - s, fq = q - qi + (g >> 1);
        if ((s < o) != (pass == 0) || (s == o && (g & 1)) || fq >= nq) continue;
        const int k = (g & 1) ? o : s;
        const float* x = lanes + r * LR + g * 8;
        float* h = wp + (size_t)(g >> 1) * NP * nz + k;
        float v[NP];
        auto sums = [&](const float* y) {
          v[0] = tree_mu<8>(y);
          if (!TAN) {
            float ax[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) ax[j] = fabsf(y[j]);
            v[1] = tree_mu<8>(ax);
            v[2] = tree_mu<8>(y + 32);
            v[3] = tree_mu<8>(y + 64);
            v[4] = tree_mu<8>(y + 96);
          }
        };
        sums(x);
        if (s < o) {
#pragma unroll
          for (int j = 0; j < NP; ++j) h[(size_t)j * nz] = v[j];
          continue;
        }
        float w[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) w[j] = s > o ? h[(size_t)j * nz] : v[j];
        if (s == o) sums(x + 8);   // the other hemisphere's lanes
        const float* fi = st + (size_t)(fl - qi + (g >> 1)) * row;
        if (TAN) {
          write_tan(cd, (size_t)k * pitch + fq, fi[3 * plane + k], add(v[0], w[0]));
        } else {
          write_base(cd, (size_t)fq * nz + k, df_make(fi[2 * plane + k], fi[3 * plane + k]), df_load(T.c2p, fq),
                     T.c2f[fq], add(v[0], w[0]), add(v[1], w[1]), add(v[2], w[2]), add(v[3], w[3]), add(v[4], w[4]));
        }
      }
      __syncwarp();
    }
  }
  if (up && m < nmu && valid && !TAN) cd.w.Iem[(size_t)q * nmu + m] = __dmul_rn((double)I, c2);
}

template <bool TAN>
__global__ void __launch_bounds__(128 * kWarpStage2) k_formal_sweep_warp(const ColDesc* __restrict__ cols) {
  extern __shared__ float s_tab[];   // [nz] |dz|, [nz] 1/|dz|, staged rows [4][F][row], per warp [2][parts][nz] and a chunk
  const ColDesc& cd = cols[blockIdx.y];
  const int mode = eval_mode_f(cd);
  if (mode == EV_SKIP || (mode == EV_TANGENT) != TAN) return;
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq;
  const int warps = blockDim.x / (32 * kWarpStage2), F = 2 * warps, qb = blockIdx.x * F;
  if (qb >= nq) return;   // uniform over the block
  float* s_dz = s_tab;
  float* s_idz = s_tab + nz;
  float* st = s_idz + nz;
  const int row = warp_row(nz);
  const size_t plane = (size_t)F * row;
  stage_dz(T, s_dz, s_idz);
  if (TAN) stage_tan(cd, qb, F, st, row);
  else stage_base(cd, mode, qb, F, st, row);
  __syncthreads();
  const int wid = threadIdx.x >> 5, fl = wid * 2 + ((threadIdx.x & 31) >> 4);
  if (wid >= warps) return;   // these warps only stage
  float* wp = st + 4 * plane + (size_t)wid * (2 * warp_parts(TAN) * nz + kWarpChunk * warp_lanes_row(TAN));
  sweep_warp<TAN>(cd, qb + fl, fl, st, row, plane, wp, s_dz, s_idz);
}

// Angle counts with their own instantiation; a launch uses the smallest one
// that covers every column of the batch (columns with fewer angles predicate
// the rest off).
static int sweep_mu_class(int nmu) {
  if (nmu <= 2) return 2;
  if (nmu <= 3) return 3;
  if (nmu <= 4) return 4;
  if (nmu <= 5) return 5;
  return 8;
}

// Dynamic shared memory of a sweep block: its |dz| tables, padded so that at
// most ``occ`` blocks fit on a multiprocessor when occ > 0. Fewer resident
// columns keep the outward pass's re-reads of the inward pass's inputs in L2.
static size_t sweep_smem(int max_nz, int occ, int threads, bool tan, bool fuse = false) {
  const size_t need =
      sizeof(float) * (2 * (size_t)max_nz + (fuse ? ring_floats(threads) : 0) + (tan ? 0 : stage_floats(threads)));
  if (occ <= 0) return need;
  const size_t cap = (size_t)227 * 1024;
  const size_t pad = (size_t)228 * 1024 / occ - 1024;
  return std::min(cap, std::max(need, pad));
}

// The packed tangent sweep of the launch's largest angle count.
static void launch_pair(const Batch& b, cudaStream_t s, size_t sm) {
  using Kernel = void (*)(const ColDesc*, float);
  static const Kernel k[kMaxMu] = {k_formal_sweep_pair<1>, k_formal_sweep_pair<2>, k_formal_sweep_pair<3>,
                                   k_formal_sweep_pair<4>, k_formal_sweep_pair<5>, k_formal_sweep_pair<6>,
                                   k_formal_sweep_pair<7>, k_formal_sweep_pair<8>};
  static_assert(kMaxMu == 8, "one instantiation per angle count");
  k[b.max_nmu - 1]<<<dim3((b.max_nq + 2 * kPairThreads - 1) / (2 * kPairThreads), b.ncols), kPairThreads, sm, s>>>(
      b.d_cols, 1.0f);
}

template <int MU>
static void launch_mu(const Batch& b, cudaStream_t s, int threads, int which, int occ_tan, int occ_base, int fuse) {
  dim3 g((b.max_nq + threads - 1) / threads, b.ncols);
  if (which != 1) {
    const size_t sm = sweep_smem(b.max_nz, occ_tan, threads, true, fuse != 0);
    if (fuse) k_formal_sweep_fused<MU><<<g, threads, sm, s>>>(b.d_cols);
    else launch_pair(b, s, sm);
  }
  if (which != 2)
    k_formal_sweep<MU><<<g, threads, sweep_smem(b.max_nz, occ_base, threads, false), s>>>(b.d_cols);
}

template <int MU>
static int allow_smem_pair() {
  JFNK_CUDA(cudaFuncSetAttribute(k_formal_sweep_pair<MU>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  if constexpr (MU > 1) return allow_smem_pair<MU - 1>();
  return JFNK_OK;
}

template <int MU>
static int allow_smem_mu() {
  JFNK_CUDA(cudaFuncSetAttribute(k_formal_sweep_fused<MU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 227 * 1024));
  JFNK_CUDA(cudaFuncSetAttribute(k_formal_sweep<MU>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  return JFNK_OK;
}

// Warps per block of the warp variant: the most whose shared memory lets three
// blocks share a multiprocessor, else one warp (0: a column too deep for it).
static int warp_size(int nz, bool tan) {
  for (int w : {4, 2})
    if (warp_variant_smem(nz, w, tan) <= (size_t)75 * 1024) return w;
  return warp_variant_smem(nz, 1, tan) <= (size_t)227 * 1024 ? 1 : 0;
}

// variant 1: ``size`` threads per block, at most occ_tan / occ_base blocks per
// SM (0: no cap); variant 2: ``size`` warps per block; which: 0 every column,
// 1 base-type evaluations, 2 tangent ones
static int launch_sweep_cfg(const Batch& b, cudaStream_t s, int variant, int size, int which = 0, int occ_tan = 0,
                            int occ_base = 0, int fuse = 0) {
  if (fuse && (variant != 1 || size != kFusedThreads))
    return fail(JFNK_E_INVALID, "fused tangent sweep: thread variant with 128-thread blocks only");
  if (variant == 2) {
    // two frequencies per warp; the warps per block follow from the depth
    auto grid = [&](int w) { return dim3((b.max_nq + 2 * w - 1) / (2 * w), b.ncols); };
    if (which != 1) {
      const int w = warp_size(b.max_nz, true);
      k_formal_sweep_warp<true><<<grid(w), 32 * w * kWarpStage2, warp_variant_smem(b.max_nz, w, true), s>>>(b.d_cols);
    }
    if (which != 2) {
      const int w = warp_size(b.max_nz, false);
      k_formal_sweep_warp<false><<<grid(w), 32 * w * kWarpStage2, warp_variant_smem(b.max_nz, w, false), s>>>(b.d_cols);
    }
  } else {
    switch (sweep_mu_class(b.max_nmu)) {
      case 2: launch_mu<2>(b, s, size, which, occ_tan, occ_base, fuse); break;
      case 3: launch_mu<3>(b, s, size, which, occ_tan, occ_base, fuse); break;
      case 4: launch_mu<4>(b, s, size, which, occ_tan, occ_base, fuse); break;
      case 5: launch_mu<5>(b, s, size, which, occ_tan, occ_base, fuse); break;
      default: launch_mu<8>(b, s, size, which, occ_tan, occ_base, fuse); break;
    }
  }
  JFNK_CUDA(cudaGetLastError());
  return JFNK_OK;
}

int sweep_prepare(Batch* b) {
  // the attribute is the kernel's, not this batch's: always the largest size
  JFNK_CUDA(cudaFuncSetAttribute(k_formal_sweep_warp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  JFNK_CUDA(cudaFuncSetAttribute(k_formal_sweep_warp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
  int rc;
  if ((rc = allow_smem_mu<2>()) || (rc = allow_smem_mu<3>()) || (rc = allow_smem_mu<4>()) ||
      (rc = allow_smem_mu<5>()) || (rc = allow_smem_mu<8>()) || (rc = allow_smem_pair<kMaxMu>()))
    return rc;
  if (b->sweep_variant == 0 && sweep_small(b->ncols, b->max_nq, b->n_sm) && sweep_warp_size(b->max_nz) > 0) {
    // nothing to tune: the variant's shape follows from the depth
    b->sweep_variant = b->tuned_variant = 2;
    b->formal_threads = b->tuned_size = sweep_warp_size(b->max_nz);
    b->optan_depths = 16;   // the separate opacity kernel's default, should a forced variant launch it
    b->tuned = true;
  }
  if (b->sweep_variant == 0) {
    b->sweep_variant = 1;
    b->formal_threads = 128;
  }
  return JFNK_OK;
}

bool sweep_fused(const Batch& b) { return b.sweep_fuse > 0 && b.sweep_variant != 2 && b.max_overlap <= kQMetaT; }

int launch_formal_sweep(const Batch& b, cudaStream_t s, int which) {
  return launch_sweep_cfg(b, s, b.sweep_variant == 2 ? 2 : 1, b.formal_threads > 0 ? b.formal_threads : 128,
                          which, b.sweep_occ, b.sweep_occ_base, sweep_fused(b) ? b.sweep_fuse : 0);
}

// Launches of fewer frequencies than these (256 per multiprocessor) take the
// warp variant: one thread per frequency would leave most warp slots empty.
bool sweep_small(int ncols, int max_nq, int n_sm) { return (long)ncols * max_nq < 256L * n_sm; }

int sweep_warp_size(int nz) { return std::min(warp_size(nz, true), warp_size(nz, false)); }

// Autotuner of a large batch, timed on its own columns: the opacity tangent's
// run of depths per thread, then a cap of resident blocks per SM for the
// tangent sweep (the columns in tangent mode) and for the base-type sweep (in
// base mode). Every choice gives bit-identical results, so it changes the speed
// only. (Block sizes of 32 to 256 threads and the warp variant were candidates
// once: 128 threads always stayed for launches of this size, and the smaller
// ones take the warp variant by rule; the first solve of a 512-column plan went
// from 990 to 650 ms without them.)
int sweep_autotune(Batch* b, cudaStream_t s) {
  cudaEvent_t e0, e1;
  JFNK_CUDA(cudaEventCreate(&e0));
  JFNK_CUDA(cudaEventCreate(&e1));
  int rc = JFNK_OK;
  // a candidate's time: the fastest of three launches timed one by one, after a
  // warm-up (single launches differ by a few per cent; the minimum is stable)
  auto timed = [&](auto launch, float* ms) -> int {
    int r = launch();   // warm-up
    if (r) return r;
    *ms = 1e30f;
    for (int i = 0; i < 3; ++i) {
      if (cudaEventRecord(e0, s) != cudaSuccess) return fail(JFNK_E_CUDA, "autotune event");
      if ((r = launch())) return r;
      float t = 0.f;
      if (cudaEventRecord(e1, s) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
          cudaEventElapsedTime(&t, e0, e1) != cudaSuccess)
        return fail(JFNK_E_CUDA, "autotune timing");
      *ms = std::min(*ms, t);
    }
    return JFNK_OK;
  };
  // the tangent sweep with the opacity-tangent launch it needs, the base-type sweep
  auto tangent = [&](int occ) {
    const int r = launch_opacity_tan(*b, s);
    return r ? r : launch_sweep_cfg(*b, s, 1, 128, 2, occ);
  };
  auto base = [&](int occ) { return launch_sweep_cfg(*b, s, 1, 128, 1, 0, occ); };
  // the opacity tangent's run of depths per thread (the depth tile of its
  // grid): the default of 16 unless another run gains 2 %
  float best = 0.f;
  int best_depths = 16;
  for (int dr : {16, 8, 32}) {
    float ms = 0.f;
    if ((rc = timed([&] { return launch_opacity_tan(*b, s, dr); }, &ms))) break;
    if (dr == 16) best = 0.98f * ms;
    else if (ms < best) { best = ms; best_depths = dr; }
  }
  b->optan_depths = best_depths;
  // The fused opacity tangent (forced variant only) is not a candidate: timed
  // alone it can win, but inside a tick the separate opacity-tangent kernel
  // overlaps the base-type chain on the other stream, and the fused sweep
  // made the whole solve about 11 % slower.
  //
  // caps of resident blocks per SM, of the tangent sweep (the columns in tangent
  // mode), then of the base-type sweep (in base mode); no cap stays unless one
  // gains 2 %: closer than that, single measurements flip between runs
  int best_occ = 0, best_base = 0;
  best = 1e30f;
  for (int occ : {0, 4}) {
    float ms = 0.f;
    if (rc || (rc = timed([&] { return tangent(occ); }, &ms))) break;
    if (occ == 0) ms *= 0.98f;
    if (ms < best) { best = ms; best_occ = occ; }
  }
  if (!rc && !(rc = batch_set_forced_mode(b, EV_BASE, s))) {
    best = 1e30f;
    for (int occ : {0, 3, 4}) {
      float ms = 0.f;
      if ((rc = timed([&] { return base(occ); }, &ms))) break;
      if (occ == 0) ms *= 0.98f;
      if (ms < best) { best = ms; best_base = occ; }
    }
    if (!rc) rc = batch_set_forced_mode(b, EV_TANGENT, s);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  b->sweep_variant = 1;
  b->formal_threads = 128;
  b->sweep_occ = best_occ;
  b->sweep_occ_base = best_base;
  b->sweep_fuse = 0;
  return JFNK_OK;
}

}  // namespace jfnk
