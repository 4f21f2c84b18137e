// FP64 evaluation of static columns in one kernel per tile of frequencies
// (steps a1 to a3: opacity, formal solution, angle and frequency integrals),
// with the formal solution's coefficients kept for the Newton step's tangents.
//
// What bounds it: GB300 issues one FP64 warp instruction per SM every 16
// cycles, so an evaluation costs the FP64 instructions of its ray-points,
// whatever else it does. Three things lower that count:
//   - a layer's coefficients e = exp(-dtau), w, a, b (App. A.1) depend on the
//     opacity of the layer and on |mu| only: one set serves the ray going out
//     through the layer and the one coming in;
//   - they do not change while n is fixed. A base evaluation leaves e, w and
//     the slope of each ray's intensity on its own dtau,
//       g = -(e D^u + bq (S^u - S^k))/(2 mu),
//     in device memory (L2 for one column), and every Jacobian-vector product
//     of that Newton step is the recurrence
//       dD^k = dD^u e + g |dz|(dchi^k + dchi^u) + w (dS^u - dS^k):
//     three FMAs per ray-point instead of an exponential and about 40 others;
//   - the ray sums take one FMA per ray and quantity, and the re-anchoring of
//     D = I - S on the better-conditioned form compares high words.
// The opacity of the tile and the rate integrals over it are formed in the
// same block (two launches and the round trips of chi, dJ and the Lambda
// diagonals fewer); a tile leaves its part of each integral it meets, and the
// assembly adds the parts in an order set by the atom (no atomics).
//
// A block takes Qb frequencies (cached_default_qb) of one column: all threads
// form the coefficients, one thread per ray runs the recurrences over chunks
// of kChunk layers (loads a batch of layers ahead), all threads add the rays
// of the chunk. Lanes run over frequencies first, so the coefficient planes
// [tile][layer][5][angle][Qb] are read in contiguous rows.
//
// Measured (kernel time, warm L2; the 8 or 10 us added the parts, now in the
// assembly), against the fused kernel with its separate opacity and rate
// kernels: 82 depths x 1,005 frequencies x 5 angles, base
// 244 + 11 + 59 -> 87 + 8 us, tangent 149 + 11 + 12 -> 26 + 8 us; 101 x 41 x 5,
// base 126 + 8 + 18 -> 50 + 10 us, tangent 48 + 8 + 11 -> 18 + 10 us. A base
// evaluation is bound by its FP64 instructions (half of it the coefficients; the
// FP64 pipe is 58 % busy over the launch, stalls are the chunks' barriers and
// shared memory), a tangent by the chain of chunks (41 %).
#include <algorithm>
#include <cmath>

#include "formal_coef.cuh"
#include "step_coef.cuh"

namespace jfnk {

constexpr int kPlanes = 5;    // e, w, P_up (later g_up), P_dn (later g_dn), bq dS
constexpr int kChunk = 8;     // layers between two ray sums
constexpr int kMaxQb = 8;
constexpr int kItems = 3;     // ray steps of a chunk per helper thread: kChunk 128 <= kItems (kEvalThreads - 128)
constexpr int kBufRows = 8 * kChunk + 2 * (2 * kChunk + 1) + kChunk;
static_assert(kChunk * 128 <= kItems * (kEvalThreads - 128), "a chunk's ray steps fit the helpers");
constexpr size_t kCachedSmem = (size_t)222 * 1024;   // beside the static shared memory

__device__ ExpEntry d_exp_tab[kExpTab];   // for neg_exp

__host__ __device__ inline int pad_qb(int qb) { return qb | 1; }   // odd row stride: no bank conflicts over depths

// Doubles shared in turn by the recurrence's buffers (two chunks of e, X, P, Y
// in, two of D, I out with the D before them, one of g) and by the level sums
// of at least 32 depths.
__host__ __device__ inline size_t chunk_doubles(int qb, int nmu, int nl) {
  const size_t rays = (size_t)kBufRows * 2 * nmu * qb, zeta = (size_t)qb * nl * 32;
  return rays > zeta ? rays : zeta;
}

size_t cached_smem_bytes(int qb, int nz, int nmu, int nl) {
  const size_t Z = (size_t)nz * pad_qb(qb);
  return sizeof(double) * (7 * Z + chunk_doubles(qb, nmu, nl)) + sizeof(int) * ((size_t)qb * kMaxT);
}

// Doubles of the coefficient planes and of the rate parts of one column.
size_t cached_planes(int qb, int nz, int nq, int nmu) {
  return (size_t)((nq + qb - 1) / qb) * (nz - 1) * kPlanes * qb * nmu;
}
size_t cached_parts(int qb, int nz, int nl, int nwin, int nt) {
  // a transition's window of nw points meets at most (nw - 1)/qb + 2 tiles
  return ((size_t)nwin / qb + 2 * (size_t)nt) * (kPartFixed + nl) * nz;
}

// Frequencies per block of a column: the smallest (waves of blocks) x (FP64
// warp instructions of a block per layer), at 2 n_mu qb/32 full warps' worth
// of about 18 (coefficients, ray sums) plus 7 per warp of rays (recurrences,
// partly filled), for the column alone on the device: 7 for 1,005 frequencies
// (144 blocks on 152 SMs), 1 for 41. It sets the order of the rate sums, so it
// must not depend on the batch: a column's result is the same alone and in any
// batch that takes the cached evaluation (batch_create: one whose planes are too
// large for it takes the fused kernel, with other roundings).
int cached_default_qb(int nq, int nz, int nmu, int nl, int n_sm) {
  int best = 0;
  double cost = 0.0;
  for (int qb = 1; qb <= kMaxQb; ++qb) {
    if (cached_smem_bytes(qb, nz, nmu, nl) > kCachedSmem || 2 * nmu * qb > 128) break;
    const long blocks = (nq + qb - 1) / qb;
    const double waves = blocks <= 4L * n_sm ? (double)((blocks + n_sm - 1) / n_sm) : (double)blocks / n_sm;
    const int rays = 2 * nmu * qb;
    const double c = waves * (18.0 * rays / 32.0 + 7.0 * ((rays + 31) / 32));
    if (!best || c < cost) {
      best = qb;
      cost = c;
    }
  }
  return best;
}

namespace {

__device__ __forceinline__ int mode_of(const ColDesc& cd) { return eval_mode_f(cd); }

__device__ __forceinline__ const double* dir_of(const ColDesc& cd) {
  if (cd.forced_mode >= 0) return cd.w.v;
  const int N = cd.t.nz * cd.t.nl;
  return cd.w.st->phase == PH_RESTART ? cd.w.x : cd.w.Vb + (size_t)cd.w.st->j * N;
}

__device__ __forceinline__ int mag(double x) { return __double2hiint(x) & 0x7fffffff; }

struct Tile {
  int qb0, nqb, Qb, Qp, R5;   // first frequency, frequencies, tile size, padded size, Qb n_mu
  int tile;
};

// The transitions active at each frequency of the tile: window point << 8 |
// lower << 4 | upper, in list order, -1 past the last.
__device__ __forceinline__ void stage_lists(const ColTables& T, const Tile& g, int* s_list) {
  const bool packed = T.max_overlap <= kQMetaT;
  for (int i = threadIdx.x; i < g.nqb * kMaxT; i += blockDim.x) {
    const int ql = i / kMaxT, j = i - ql * kMaxT, q = g.qb0 + ql;
    int m = -1;
    if (packed) {
      if (j < kQMetaT) m = __ldg(T.qmeta + (size_t)j * T.nq + q);
    } else if (T.q_off[q] + j < T.q_off[q + 1]) {
      const int s = T.q_off[q] + j;
      const int t = T.q_t[s];
      m = ((T.t_base[t] + q - T.t_q0[t]) << 8) | (T.t_lo[t] << 4) | T.t_up[t];
    }
    s_list[i] = m;
  }
}

// sum V x_lo and sum g V x_up over the transitions active at a frequency (list
// L), at depth k: the loads of two transitions are issued together.
__device__ __forceinline__ void line_sums(const ColTables& T, const int* L, int k, const double* __restrict__ x,
                                          double& sl, double& su) {
  sl = su = 0.0;
  const double* xk = x + (size_t)k * T.nl;
  for (int j = 0; j < kMaxT; j += 2) {
    const int m0 = L[j], m1 = L[j + 1];
    if (m0 < 0) break;
    const size_t p0 = (size_t)(m0 >> 8) * T.nz + k, p1 = (size_t)((m1 < 0 ? m0 : m1) >> 8) * T.nz + k;
    const double v0 = T.V[p0], g0 = T.gV[p0], v1 = T.V[p1], g1 = T.gV[p1];
    const double l0 = xk[(m0 >> 4) & 15], u0 = xk[m0 & 15];
    const double l1 = xk[(m1 < 0 ? m0 : m1) >> 4 & 15], u1 = xk[(m1 < 0 ? m0 : m1) & 15];
    sl = fma(v0, l0, sl);
    su = fma(g0, u0, su);
    if (m1 < 0) break;
    sl = fma(v1, l1, sl);
    su = fma(g1, u1, su);
  }
}

// Parts of the rate integrals of transition t at depth k over the tile's
// frequencies: sum W V J and sum W g V J (J: dJ in tangent evaluations).
__device__ __forceinline__ void rate_parts(const ColTables& T, const Tile& g, int t, int k, const double* s_J,
                                           double* part) {
  const int q0 = T.t_q0[t], qa = max(q0, g.qb0), n = min(T.t_q1[t], g.qb0 + g.nqb - 1) - qa + 1;
  const size_t pk = (size_t)(T.t_base[t] + qa - q0) * T.nz + k;
  double wv[kMaxQb], wg[kMaxQb];
#pragma unroll
  for (int i = 0; i < kMaxQb; ++i) {
    const size_t p = pk + (size_t)min(i, n - 1) * T.nz;
    wv[i] = T.WV[p];
    wg[i] = T.WgV[p];
  }
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int i = 0; i < kMaxQb; ++i)
    if (i < n) {
      const double J = s_J[k * g.Qp + qa - g.qb0 + i];
      a0 = fma(wv[i], J, a0);
      a1 = fma(wg[i], J, a1);
    }
  part[k] = a0;
  part[T.nz + k] = a1;
}

// Barrier of the threads from ``first`` on (the warps without rays).
__device__ __forceinline__ void helper_sync(int first) {
  asm volatile("bar.sync 1, %0;" ::"r"((int)blockDim.x - first) : "memory");
}

}  // namespace

// One F-class evaluation of one tile of frequencies (grid: tiles x columns).
//
// Each SM sub-partition starts an FP64 warp instruction every 64 cycles, so a
// warp that carries rays must do little else: the first warps (one lane per
// ray) run the recurrences alone, D' = D e + X and I' = I e + P, over chunks of
// kChunk layers, while the others form e, X, P of the next chunk in shared
// memory (from planes loaded a chunk before) and add the rays of the previous
// one. One block barrier per chunk.
// MU: angles of every column of the launch (0: read from the column).
template <int MU>
__global__ void __launch_bounds__(kEvalThreads) k_eval64(const ColDesc* __restrict__ cols, const SolverOpts* bopts) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double s_inv2mu[kMaxMu], s_hw[kMaxMu], s_2mu[kMaxMu];
  __shared__ ExpEntry s_tab[kExpTab];
  __shared__ int s_act[kMaxT], s_off[kMaxT], s_nact;
  const ColDesc& cd = cols[blockIdx.y];
  const int mode = mode_of(cd);
  if (mode == EV_SKIP) return;
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq, nmu = MU ? MU : T.nmu, nl = T.nl, Qb = cd.w.cq;
  Tile g;
  g.tile = blockIdx.x;
  g.Qb = Qb;
  g.qb0 = g.tile * Qb;
  if (g.qb0 >= nq) return;
  g.nqb = min(Qb, nq - g.qb0);
  g.Qp = pad_qb(Qb);
  g.R5 = Qb * nmu;
  const int Qp = g.Qp, nqb = g.nqb, qb0 = g.qb0, R5 = g.R5;
  const int nray = 2 * R5;
  const size_t Z = (size_t)nz * Qp;
  double* s_S = sm;               // S^k
  double* s_chi = s_S + Z;        // chi^k; then sum w I; then J
  double* s_tz = s_chi + Z;       // sum w D; then Lambda_chi
  double* s_rs = s_tz + Z;        // sum w |D|
  double* s_dS = s_rs + Z;        // S^{k+1} - S^k; then Lambda_eta
  double* s_A = s_dS + Z;         // per layer, sum over the angles of w a
  double* s_G = s_A + Z;          // sum of w dI/dchi without the local term
  double* s_buf = s_G + Z;        // the recurrence's chunks; then the level sums
  double* s_in = s_buf;                               // [2][4][kChunk][nray]: e, X, P, Y
  double* s_out = s_buf + (size_t)8 * kChunk * nray;  // [2][2 kChunk + 1][nray]: D before the chunk, D, I
  double* s_g = s_out + (size_t)2 * (2 * kChunk + 1) * nray;   // [kChunk][nray]: g
  int* s_list = reinterpret_cast<int*>(s_buf + chunk_doubles(Qb, nmu, nl));
  double* cf = cd.w.cf + (size_t)g.tile * (nz - 1) * kPlanes * R5;
  const bool tan = (mode == EV_TANGENT), der = (mode == EV_BASE || mode == EV_RH92), base = (mode == EV_BASE);

  stage_lists(T, g, s_list);
  for (int m = threadIdx.x; m < nmu; m += blockDim.x) {
    const Ang64 a = T.ang64[m];
    s_inv2mu[m] = a.inv2mu;
    s_hw[m] = a.hw;
    s_2mu[m] = a.two_mu;
  }
  if (!tan)
    for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) s_tab[i] = d_exp_tab[i];
  if (threadIdx.x < 32) {
    // the transitions whose windows meet the tile, and their part slots
    int tile0, ntile;
    const int off = part_offset(T, Qb, threadIdx.x, tile0, ntile);
    const bool on = g.tile >= tile0 && g.tile < tile0 + ntile;
    const unsigned b = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int i = __popc(b & ((1u << threadIdx.x) - 1));
      s_act[i] = threadIdx.x;
      s_off[i] = off + g.tile - tile0;
    }
    if (threadIdx.x == 0) s_nact = __popc(b);
  }
  __syncthreads();
  const int nslot = kPartFixed + nl;

  // this thread's ray, or its place among the warps without rays
  const int ray = threadIdx.x;
  const int hfirst = (nray + 31) & ~31;   // first helper thread (2 n_mu Qb <= 128)
  const bool up = ray >= R5;
  const int rr = up ? ray - R5 : ray;
  const int rm = rr / Qb, rq = rr - rm * Qb;
  const bool run = ray < nray && rq < nqb, helper = (int)threadIdx.x >= hfirst;
  const int nch = (nz - 2) / kChunk + 1;   // chunks of the nz - 1 layers
  // this helper's ray steps of every chunk: their row, layer and planes in chunk 0
  const int t0 = threadIdx.x - hfirst, nh = blockDim.x - hfirst;
  int ir[kItems], il[kItems];
  double* ip[kItems];
  double be[kItems], bw[kItems], bp[kItems], by[kItems];
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = t0 + j * nh, r = i / nray, y = i - r * nray;
    const bool u = y >= R5;
    const int yr = u ? y - R5 : y;
    ir[j] = !helper || r >= kChunk || yr % Qb >= nqb ? nz : r;   // nz: never
    il[j] = u ? nz - 2 - r : r;
    ip[j] = cf + (ptrdiff_t)il[j] * kPlanes * R5 + yr;
  }
  // this helper's place in the ray sums of every chunk: hemisphere, row and
  // frequency (the last warps take them, the first ones carry more ray steps)
  const int si = nh - 1 - t0, sh = si / (kChunk * Qb), sr = (si - sh * kChunk * Qb) / Qb, sq = si % Qb;
  const bool sums = helper && sh < 2 && sq < nqb;
  auto item_up = [&](int j) { return t0 + j * nh - ir[j] * nray >= R5; };
  // the planes of chunk c, into registers
  auto load = [&](int c) {
#pragma unroll
    for (int j = 0; j < kItems; ++j)
      if (c * kChunk + ir[j] < nz - 1) {
        const bool u = item_up(j);
        const double* p = ip[j] + (u ? -1 : 1) * (ptrdiff_t)c * kChunk * kPlanes * R5;
        be[j] = p[0];
        bw[j] = p[R5];
        if (tan || der) bp[j] = p[(u ? 2 : 3) * R5];
        if (base) by[j] = p[4 * R5];
      }
  };
  // the inputs of chunk c, from registers into its buffer
  auto store = [&](int c) {
    double* in = s_in + (size_t)(c & 1) * 4 * kChunk * nray;
#pragma unroll
    for (int j = 0; j < kItems; ++j)
      if (c * kChunk + ir[j] < nz - 1) {
        const bool u = item_up(j);
        const int i = t0 + j * nh, l = il[j] + (u ? -c * kChunk : c * kChunk);
        const int e = l * Qp + (u ? i - ir[j] * nray - R5 : i - ir[j] * nray) % Qb;
        const double x = bw[j] * s_dS[e];
        in[i] = be[j];
        if (tan) {
          // s_dS: dS^{k+1} - dS^k, s_tz: |dz|(dchi^k + dchi^{k+1})
          in[kChunk * nray + i] = fma(bp[j], s_tz[e], u ? x : -x);
        } else {
          in[kChunk * nray + i] = u ? x : -x;
          if (der) in[2 * kChunk * nray + i] = bp[j];
          if (base) in[3 * kChunk * nray + i] = by[j];
        }
      }
  };

  if (tan) {
    load(0);   // the base evaluation's planes, while the opacity's tangent is formed
    double* s_dc = s_S;      // dchi^k; then dJ
    double* s_dT = s_chi;    // dS^k
    double* s_acc = s_rs;    // sum over the rays of w dD
    const double* v = dir_of(cd);
    const double* rchi = reinterpret_cast<const double*>(cd.w.chi);
    for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
      const int ql = i / nz, k = i - ql * nz;
      const size_t o = (size_t)(qb0 + ql) * nz + k;
      const double S = cd.w.S[o], rc = rchi[o];
      double dl, de;
      line_sums(T, s_list + ql * kMaxT, k, v, dl, de);
      const double dc = dl - de;
      s_dc[k * Qp + ql] = dc;
      s_dT[k * Qp + ql] = fma(-S, dc, de) * rc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
      const int k = i / nqb, ql = i - k * nqb, e = k * Qp + ql;
      // the boundary rays start from dD = -dS at the bottom (outgoing) and the top (ingoing)
      double acc = 0.0;
      if (k == 0 || k == nz - 1)
        for (int m = 0; m < nmu; ++m) acc = fma(-s_hw[m], s_dT[e], acc);
      s_acc[e] = acc;
      if (k < nz - 1) {
        s_tz[e] = T.dz[k] * (s_dc[e] + s_dc[e + Qp]);
        s_dS[e] = s_dT[e + Qp] - s_dT[e];
      }
    }
    __syncthreads();
    store(0);
    load(1);
    double dD = run ? -s_dT[(up ? nz - 1 : 0) * Qp + rq] : 0.0;
    __syncthreads();
    for (int c = 0; c <= nch; ++c) {
      if (!helper) {
        if (c < nch && run) {
          const int rows = min(kChunk, nz - 1 - c * kChunk);
          const double* in = s_in + (size_t)(c & 1) * 4 * kChunk * nray + ray;
          double* out = s_out + (size_t)(c & 1) * (2 * kChunk + 1) * nray + ray;
          double e[kChunk], X[kChunk];
#pragma unroll
          for (int r = 0; r < kChunk; ++r) {
            const int q = min(r, rows - 1) * nray;
            e[r] = in[q];
            X[r] = in[kChunk * nray + q];
          }
#pragma unroll
          for (int r = 0; r < kChunk; ++r) X[r] = dD = r < rows ? fma(dD, e[r], X[r]) : dD;
#pragma unroll
          for (int r = 0; r < kChunk; ++r)
            if (r < rows) out[r * nray] = X[r];
        }
      } else {
        if (c > 0) {
          const int c0 = (c - 1) * kChunk, rows = min(kChunk, nz - 1 - c0);
          const double* out = s_out + (size_t)((c - 1) & 1) * (2 * kChunk + 1) * nray;
          // a depth can be reached by both hemispheres in one chunk (the middle
          // of the column): its two sums are then added one after the other
          const bool apart = c0 + rows < nz - 1 - c0 - rows || c0 + 1 > nz - 2 - c0;
          for (int h = 0; h < (apart ? 1 : 2); ++h) {
            if (sums && sr < rows && (apart || h == sh)) {
              const int e = (sh ? nz - 2 - (c0 + sr) : c0 + sr + 1) * Qp + sq;
              const double* x = out + sr * nray + sh * R5 + sq;
              double a = s_acc[e];
#pragma unroll
              for (int m = 0; m < nmu; ++m) a = fma(s_hw[m], x[m * Qb], a);
              s_acc[e] = a;
            }
            if (!apart) helper_sync(hfirst);
          }
        }
        if (c + 1 < nch) {
          store(c + 1);
          load(c + 2);
        }
      }
      __syncthreads();
    }
    for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
      const int k = i / nqb, ql = i - k * nqb, e = k * Qp + ql;
      s_dc[e] = (s_dT[e] + s_acc[e]) * T.c2[qb0 + ql];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < s_nact * nz; i += blockDim.x) {
      const int a = i / nz, k = i - a * nz;
      rate_parts(T, g, s_act[a], k, s_dc, cd.w.rpart + (size_t)s_off[a] * nslot * nz);
    }
    return;
  }

  // ---- values: opacity and source function (Eqs. chi, eta) ------------------
  const double* n = eval_pops(cd, mode);
  const double* Jd = jdag_ptr(cd);
  for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
    const int ql = i / nz, k = i - ql * nz;
    const size_t o = (size_t)(qb0 + ql) * nz + k;
    const double sca = T.chi_sca[k], chib = T.chi_c[o] + sca;
    const double eta_bg = T.eta_c[o] + sca * Jd[o];
    const double c2 = T.c2[qb0 + ql];
    double chl, el;
    line_sums(T, s_list + ql * kMaxT, k, n, chl, el);
    const double chi = chib + (chl - el), eta = fma(c2, el, eta_bg);
    // S = eta/(chi 2 h nu^3/c^2), rounded once (quotient plus its remainder)
    const double d = chi * c2, rd = 1.0 / d, q0 = eta * rd, S = fma(fma(-q0, d, eta), rd, q0), rc = c2 * rd;
    s_chi[k * Qp + ql] = chi;
    s_S[k * Qp + ql] = S;
    s_A[k * Qp + ql] = 0.0;
    if (der) {
      reinterpret_cast<double*>(cd.w.chi)[o] = rc;   // 1/chi: all that later steps need
      cd.w.S[o] = S;
      if (mode == EV_RH92) cd.w.eta[o] = eta;
    }
  }
  __syncthreads();
  // ---- coefficients of every (layer, angle), for both hemispheres ------------
  for (int i = threadIdx.x; i < nqb * (nz - 1); i += blockDim.x) {
    const int l = i / nqb, ql = i - l * nqb, e0 = l * Qp + ql;
    const double tz = T.dz[l] * (s_chi[e0] + s_chi[e0 + Qp]), rs = 1.0 / tz;
    const double S0 = s_S[e0], S1 = s_S[e0 + Qp], dS = S1 - S0;
    s_dS[e0] = dS;
    double* c = cf + (size_t)l * kPlanes * R5 + ql;
    double A = 0.0;
#pragma unroll
    for (int m = 0; m < nmu; ++m, c += Qb) {
      const double x = tz * s_inv2mu[m];
      double e, w, a, bq, om;
      step_coef(x, rs * s_2mu[m], s_tab, e, w, a, bq, om);
      c[0] = e;
      c[R5] = w;
      if (der) {
        // outgoing a S^k + b S^{k+1}, ingoing a S^{k+1} + b S^k, b = bq x = om - a
        const double Y = bq * dS, yx = Y * x;
        c[2 * R5] = fma(om, S0, yx);
        c[3 * R5] = fma(om, S1, -yx);
        c[4 * R5] = Y;
        A = fma(s_hw[m], a, A);
      }
    }
    s_A[e0] = A;
  }
  // ---- recurrences ------------------------------------------------------------
  __syncthreads();
  double* s_I = s_chi;
  double* s_D = s_tz;
  double* s_aD = s_rs;
  double* s_Le = s_dS;
  for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
    const int k = i / nqb, ql = i - k * nqb, e = k * Qp + ql;
    double d = 0.0, in = 0.0, ad = 0.0;
    if (k == 0 || k == nz - 1) {
      const double Ib = k == 0 ? 0.0 : T.Bn[(size_t)(qb0 + ql) * nz + nz - 1] / T.c2[qb0 + ql];
      const double D = Ib - s_S[e];
      for (int m = 0; m < nmu; ++m) {
        d = fma(s_hw[m], D, d);
        ad = fma(s_hw[m], fabs(D), ad);
        in = fma(s_hw[m], Ib, in);
      }
    }
    s_I[e] = in;
    s_D[e] = d;
    s_aD[e] = ad;
    s_G[e] = 0.0;
  }
  double D = 0.0, I = 0.0;
  int M = 0;   // exponent word of the attenuated bound of |D| upstream
  if (run) {
    I = up ? T.Bn[(size_t)(qb0 + rq) * nz + nz - 1] / T.c2[qb0 + rq] : 0.0;
    D = I - s_S[(up ? nz - 1 : 0) * Qp + rq];
    M = mag(D);
  }
  load(0);
  store(0);
  load(1);
  __syncthreads();
  for (int c = 0; c <= nch; ++c) {
    if (!helper) {
      if (c < nch && run) {
        const int c0 = c * kChunk, rows = min(kChunk, nz - 1 - c0);
        const double* in = s_in + (size_t)(c & 1) * 4 * kChunk * nray + ray;
        double* out = s_out + (size_t)(c & 1) * (2 * kChunk + 1) * nray + ray;   // D before, D after each step, I
        out[0] = D;
        double e[kChunk], X[kChunk], P[kChunk], Sk[kChunk];
#pragma unroll
        for (int r = 0; r < kChunk; ++r) {
          const int rq_ = min(r, rows - 1), q = rq_ * nray;
          e[r] = in[q];
          X[r] = in[kChunk * nray + q];
          if (der) {
            P[r] = in[2 * kChunk * nray + q];
            Sk[r] = s_S[(up ? nz - 2 - c0 - rq_ : c0 + rq_ + 1) * Qp + rq];
          }
        }
#pragma unroll
        for (int r = 0; r < kChunk; ++r)
          if (r < rows) {
            double Dn = fma(D, e[r], X[r]);
            if (der) {
              I = fma(I, e[r], P[r]);
              // D carries an absolute error of the order of the largest |D| met
              // upstream (attenuated), I - S one of the order of |I| + |S|: take the
              // better-conditioned form. Both bounds are kept as high words: the
              // larger of |I| and |S| for their sum, and words added for the product
              // M e, which is at most 11 % short a step (Mitchell, IRE Trans. EC-11,
              // 512, 1962). Over 4,000 random rays the largest error of D, in units of
              // the rounding of |I| + |S|, is 7.9 with these bounds, 7.3 with FP64 ones.
              M = max(M + (__double2hiint(e[r]) - 0x3ff00000), mag(Dn));
              const int anchor = max(mag(I), mag(Sk[r]));
              if (anchor < M) {
                Dn = I - Sk[r];
                M = anchor;
              }
              P[r] = I;
            }
            X[r] = D = Dn;
          }
#pragma unroll
        for (int r = 0; r < kChunk; ++r)
          if (r < rows) {
            out[(r + 1) * nray] = X[r];
            if (der) out[(kChunk + 1 + r) * nray] = P[r];
          }
      }
    } else {
      if (base && c > 0) {
        // the slope of each ray's intensity on its dtau, kept for the tangents
        const double* in = s_in + (size_t)((c - 1) & 1) * 4 * kChunk * nray;
        const double* out = s_out + (size_t)((c - 1) & 1) * (2 * kChunk + 1) * nray;
#pragma unroll
        for (int j = 0; j < kItems; ++j)
          if ((c - 1) * kChunk + ir[j] < nz - 1) {
            const bool u = item_up(j);
            const int i = t0 + j * nh;
            const double Y = in[3 * kChunk * nray + i];
            const int yr = u ? i - ir[j] * nray - R5 : i - ir[j] * nray;
            const double gm = -s_inv2mu[yr / Qb] * fma(in[i], out[i], u ? Y : -Y);
            ip[j][(u ? -1 : 1) * (ptrdiff_t)(c - 1) * kChunk * kPlanes * R5 + (u ? 2 : 3) * R5] = gm;
            s_g[i] = gm;
          }
      }
      if (c + 1 < nch) {   // into the buffer whose e, Y this thread has just read
        store(c + 1);
        load(c + 2);
      }
      if (base) helper_sync(hfirst);
      if (c > 0) {
        const int c0 = (c - 1) * kChunk, rows = min(kChunk, nz - 1 - c0);
        const double* out = s_out + (size_t)((c - 1) & 1) * (2 * kChunk + 1) * nray;
        const bool apart = c0 + rows < nz - 1 - c0 - rows || c0 + 1 > nz - 2 - c0;   // as above
        for (int h = 0; h < (apart ? 1 : 2); ++h) {
          if (sums && sr < rows && (apart || h == sh)) {
            const int k = sh ? nz - 2 - (c0 + sr) : c0 + sr + 1, l = sh ? k : k - 1;
            const int y = sr * nray + sh * R5 + sq, e = k * Qp + sq;
            double d = s_D[e], in = s_I[e], ad = s_aD[e], gs = 0.0;
#pragma unroll
            for (int m = 0; m < nmu; ++m) {
              const double hw = s_hw[m], Dk = out[nray + y + m * Qb];
              d = fma(hw, Dk, d);
              if (der) {
                ad = fma(hw, fabs(Dk), ad);
                in = fma(hw, out[(kChunk + 1) * nray + y + m * Qb], in);
                if (base) gs = fma(hw, s_g[y + m * Qb], gs);
              }
            }
            s_D[e] = d;
            if (der) {
              s_aD[e] = ad;
              s_I[e] = in;
              if (base) s_G[e] = fma(T.dz[l], gs, s_G[e]);
            }
          }
          if (!apart) helper_sync(hfirst);
        }
      }
    }
    __syncthreads();
  }
  if (run && up && der) cd.w.Iem[(size_t)(qb0 + rq) * nmu + rm] = I * T.c2[qb0 + rq];

  // ---- J and the Lambda diagonals (App. A.2 with S^u - I^u = -D^u) ------------
  for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
    const int ql = i / nz, k = i - ql * nz, e = k * Qp + ql;
    const size_t o = (size_t)(qb0 + ql) * nz + k;
    const double c2 = T.c2[qb0 + ql], S = s_S[e];
    double J = (S + s_D[e]) * c2, Lx = 0.0, Le = 0.0;
    if (der) {
      // the representation with the smaller rounding error (intensities are >= 0)
      if (fabs(s_I[e]) < s_aD[e]) J = s_I[e] * c2;
      const double rc = reinterpret_cast<const double*>(cd.w.chi)[o];
      const double A = (k < nz - 1 ? s_A[e] : 0.0) + (k > 0 ? s_A[e - Qp] : 0.0);
      Le = rc * A;
      jnew_ptr(cd)[o] = J;
      if (base) {
        Lx = fma(-S, Le, s_G[e]) * c2;
        cd.w.Lchi[o] = Lx;
        cd.w.Leta[o] = Le;
      }
    }
    s_I[e] = J;
    s_D[e] = Lx;
    s_Le[e] = Le;
  }
  __syncthreads();

  // ---- rate integrals over the tile (Eqs. Rij, Rji) ---------------------------
  if (!der) {
    for (int i = threadIdx.x; i < s_nact * nz; i += blockDim.x) {
      const int a = i / nz, k = i - a * nz;
      rate_parts(T, g, s_act[a], k, s_I, cd.w.rpart + (size_t)s_off[a] * nslot * nz);
    }
    return;
  }
  // with the preconditioner sums sum_nu W chi_t zeta_j (Sect. 2.5.1),
  // zeta_j = beta_j Lchi + gamma_j Leta, or the RH92 sums with
  // zeta_j = Psi* sum_{s: up = j} 2 h nu^3/c^2 g_s V_s: zeta is formed once per
  // (nu, depth) and level, as many depths at a time as the buffer holds
  const int pv = base ? precond_variant(cd, bopts) : 1;
  const int kt = min(nz, (int)(chunk_doubles(Qb, nmu, nl) / ((size_t)Qb * nl)));
  double* s_z = s_buf;   // [Qb][nl][kt]
  for (int k0 = 0; k0 < nz; k0 += kt) {
    const int nk = min(kt, nz - k0);
    for (int i = threadIdx.x; i < nqb * nk; i += blockDim.x) {
      const int ql = i / nk, kk = i - ql * nk, k = k0 + kk, e = k * Qp + ql;
      double* z = s_z + (size_t)ql * nl * kt + kk;
      const double Lx = s_D[e], Le = s_Le[e], c2 = T.c2[qb0 + ql], sca = T.chi_sca[k];
      for (int j = 0; j < nl; ++j)
        z[j * kt] = (pv == 2) ? sca * Le * cd.w.dJdn[((size_t)(qb0 + ql) * nz + k) * nl + j] : 0.0;
      const double cu = base ? fma(c2, Le, -Lx) : c2 * Le;
      const int* L = s_list + ql * kMaxT;
      for (int j = 0; j < kMaxT; ++j) {
        const int m = L[j];
        if (m < 0) break;
        const size_t p = (size_t)(m >> 8) * nz + k;
        if (base) {
          double& zl = z[((m >> 4) & 15) * kt];
          zl = fma(T.V[p], Lx, zl);
        }
        double& zu = z[(m & 15) * kt];
        zu = fma(T.gV[p], cu, zu);
      }
      if (pv == 3) {
        const double f = 1.0 / (1.0 - sca * Le);
        for (int j = 0; j < nl; ++j) z[j * kt] *= f;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < s_nact * nk; i += blockDim.x) {
      const int a = i / nk, kk = i - a * nk, k = k0 + kk, t = s_act[a];
      const int q0 = T.t_q0[t], qa = max(q0, qb0), nw = min(T.t_q1[t], qb0 + nqb - 1) - qa + 1;
      const double nlo = n[k * nl + T.t_lo[t]], nup = n[k * nl + T.t_up[t]];
      const size_t pk = (size_t)(T.t_base[t] + qa - q0) * nz + k;
      double wv[kMaxQb], wg[kMaxQb];
#pragma unroll
      for (int q = 0; q < kMaxQb; ++q) {
        const size_t p = pk + (size_t)min(q, nw - 1) * nz;
        wv[q] = T.WV[p];
        wg[q] = T.WgV[p];
      }
      double* part = cd.w.rpart + (size_t)s_off[a] * nslot * nz + k;
      double a0 = 0.0, a1 = 0.0, r0 = 0.0, r1 = 0.0, r3 = 0.0;
#pragma unroll
      for (int q = 0; q < kMaxQb; ++q)
        if (q < nw) {
          const int e = k * Qp + qa - qb0 + q;
          const double J = s_I[e];
          a0 = fma(wv[q], J, a0);
          a1 = fma(wg[q], J, a1);
          const double Wc = fma(wv[q], nlo, -wg[q] * nup);   // W chi_t
          if (!base) {
            const size_t o = (size_t)(qa + q) * nz + k;
            const double Le = s_Le[e], Je = fma(-Le, cd.w.eta[o], J);   // Jeff = J - Psi* eta
            r0 = fma(wv[q], Je, r0);
            r1 = fma(wg[q], Je, r1);
            r3 = fma(Wc * Le, T.eta_c[o] + T.chi_sca[k] * Jd[o], r3);
          }
          wv[q] = Wc;
        }
      part[0] = a0;
      part[nz] = a1;
      if (!base) {
        part[2 * (size_t)nz] = r0;
        part[3 * (size_t)nz] = r1;
        part[4 * (size_t)nz] = r3;
      }
      const double* z = s_z + (size_t)(qa - qb0) * nl * kt + kk;
      part += (size_t)(base ? 2 : kPartFixed) * nz;
      for (int j = 0; j < nl; ++j, z += kt, part += nz) {
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < kMaxQb; ++q)
          if (q < nw) acc = fma(wv[q], z[q * nl * kt], acc);
        part[0] = acc;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Moving columns (velocity.cu has the equations): the same evaluation with an
// opacity and a source function per ray. Nothing is shared by the hemispheres,
// so every (ray, layer) has its own coefficients; a base evaluation keeps e, h a,
// h b and h |dz|/(2 mu) G of each, h = w_mu/2, G the slope of the ray's intensity
// on its optical depth,
//   G = -I^u e + (b/dtau) S^k + (e - b/dtau) S^u   (da = (b/dtau) ddtau, db = (e - b/dtau) ddtau),
// and a product is h dI^k = h dI^u e + [h |dz|/(2 mu) G](dchi^k + dchi^u) + h a dS^k
// + h b dS^u: five FP64 instructions per ray-point besides its opacity's tangent.
// The local derivatives of the block-Jacobi sums follow from the same numbers,
// dI^k/dchi^k = |dz|/(2 mu) G - (S^k/chi^k) a, dI^k/deta^k = a/chi^k.
//
// Rays stay in shared memory over all depths ([depth][ray]); a column too deep
// for that takes the separate kernels of velocity.cu. 82 depths x 1,005
// frequencies x 10 rays: product 35 + 197 + 37 -> 76 us, base evaluation 41 +
// 245 + 8 + 205 -> 286 us.
// ---------------------------------------------------------------------------
constexpr int kMvPlanes = 4;   // e, h a, h b, then h bq and finally the slope

__host__ __device__ inline size_t mv_rows(int nz) { return 3 * (size_t)nz + 4 * kChunk; }

size_t moving_smem_bytes(int qb, int nz, int nmu) {
  return sizeof(double) * mv_rows(nz) * ((2 * nmu * qb) | 1) + sizeof(int) * ((size_t)qb * kMaxT);
}
size_t moving_planes(int qb, int nz, int nq, int nmu) {
  return (size_t)((nq + qb - 1) / qb) * (nz - 1) * kMvPlanes * 2 * nmu * qb;
}

// Frequencies per block of a moving column (0: too deep), as cached_default_qb:
// about 25 full warps' worth of FP64 instructions per ray step besides the ray
// warps' own.
int moving_default_qb(int nq, int nz, int nmu, int n_sm) {
  int best = 0;
  double cost = 0.0;
  for (int qb = 1; qb <= kMaxQb; ++qb) {
    if (moving_smem_bytes(qb, nz, nmu) > kCachedSmem || 2 * nmu * qb > 128) break;
    const long blocks = (nq + qb - 1) / qb;
    const double waves = blocks <= 4L * n_sm ? (double)((blocks + n_sm - 1) / n_sm) : (double)blocks / n_sm;
    const int rays = 2 * nmu * qb;
    const double c = waves * (25.0 * rays / 32.0 + (rays + 31) / 32);
    if (!best || c < cost) {
      best = qb;
      cost = c;
    }
  }
  return best;
}

template <int MU>
__global__ void __launch_bounds__(kEvalThreads) k_eval64_moving(const ColDesc* __restrict__ cols) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double s_inv2mu[kMaxMu], s_hw[kMaxMu];
  __shared__ ExpEntry s_tab[kExpTab];
  __shared__ int s_act[kMaxT], s_off[kMaxT], s_nact;
  const ColDesc& cd = cols[blockIdx.y];
  const int mode = mode_of(cd);
  if (mode == EV_SKIP || mode == EV_RH92) return;   // RH92 is rejected for moving columns
  const ColTables& T = cd.t;
  const int nz = T.nz, nq = T.nq, nmu = MU ? MU : T.nmu, nl = T.nl, Qb = cd.w.cq;
  Tile g;
  g.tile = blockIdx.x;
  g.Qb = Qb;
  g.qb0 = g.tile * Qb;
  if (g.qb0 >= nq) return;
  g.nqb = min(Qb, nq - g.qb0);
  g.Qp = pad_qb(Qb);
  g.R5 = Qb * nmu;
  const int nqb = g.nqb, qb0 = g.qb0, R5 = g.R5, nray = 2 * R5, rp = nray | 1;
  double* s0 = sm;                      // [nz][rp] chi (or its tangent); then dI/dchi
  double* s1 = s0 + (size_t)nz * rp;    // S (or its tangent); then dI/deta
  double* sI = s1 + (size_t)nz * rp;    // h I (or h dI)
  double* s_in = sI + (size_t)nz * rp;  // [2][2][kChunk][nray]: e, X of a chunk
  int* s_list = reinterpret_cast<int*>(sm + mv_rows(nz) * rp);
  double* cf = cd.w.cf + (size_t)g.tile * (nz - 1) * kMvPlanes * nray;
  const bool tan = (mode == EV_TANGENT), base = (mode == EV_BASE);
  const double* Vd = T.Vd ? T.Vd : T.V;                       // a static column of the batch: one profile
  const size_t dstride = T.Vd ? (size_t)T.nwin * nz : 0, per = (size_t)nq * nz;

  stage_lists(T, g, s_list);
  for (int m = threadIdx.x; m < nmu; m += blockDim.x) {
    s_inv2mu[m] = T.ang64[m].inv2mu;
    s_hw[m] = T.ang64[m].hw;
  }
  if (!tan)
    for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) s_tab[i] = d_exp_tab[i];
  if (threadIdx.x < 32) {
    int tile0, ntile;
    const int off = part_offset(T, Qb, threadIdx.x, tile0, ntile);
    const bool on = g.tile >= tile0 && g.tile < tile0 + ntile;
    const unsigned b = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int i = __popc(b & ((1u << threadIdx.x) - 1));
      s_act[i] = threadIdx.x;
      s_off[i] = off + g.tile - tile0;
    }
    if (threadIdx.x == 0) s_nact = __popc(b);
  }
  // rays: ingoing first, then outgoing, each [angle][frequency]; direction d of
  // the tables counts the outgoing ones first
  const int ray = threadIdx.x, hfirst = (nray + 31) & ~31;
  const bool up = ray >= R5;
  const int rr = up ? ray - R5 : ray, rm = rr / Qb, rq = rr - rm * Qb;
  const bool run = ray < nray && rq < nqb, helper = (int)threadIdx.x >= hfirst;
  const int t0 = threadIdx.x - hfirst, nh = blockDim.x - hfirst;
  const int nch = (nz - 2) / kChunk + 1;
  int ir[kItems], iy[kItems];
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = t0 + j * nh, r = i / nray;
    iy[j] = i - r * nray;
    ir[j] = !helper || r >= kChunk || (iy[j] >= R5 ? iy[j] - R5 : iy[j]) % Qb >= nqb ? nz : r;   // nz: never
  }
  double be[kItems], ba[kItems], bb[kItems], bg[kItems];
  auto load = [&](int c) {
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int s = c * kChunk + ir[j];
      if (s < nz - 1) {
        const double* p = cf + (size_t)(iy[j] >= R5 ? nz - 2 - s : s) * kMvPlanes * nray + iy[j];
        be[j] = p[0];
        ba[j] = p[nray];
        bb[j] = p[2 * nray];
        if (tan) bg[j] = p[3 * nray];
      }
    }
  };
  auto store = [&](int c) {
    double* in = s_in + (size_t)(c & 1) * 2 * kChunk * nray;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int s = c * kChunk + ir[j];
      if (s < nz - 1) {
        const bool u = iy[j] >= R5;
        const int k = u ? nz - 2 - s : s + 1, ku = u ? k + 1 : k - 1;
        const int e = k * rp + iy[j], eu = ku * rp + iy[j];
        double X = fma(ba[j], s1[e], bb[j] * s1[eu]);   // h (a S^k + b S^u), or of the tangents
        if (tan) X = fma(bg[j], s0[e] + s0[eu], X);
        in[ir[j] * nray + iy[j]] = be[j];
        in[(kChunk + ir[j]) * nray + iy[j]] = X;
      }
    }
  };
  if (tan) load(0);
  __syncthreads();
  const int nslot = kPartFixed + nl;

  // ---- opacity and source function of every ray, or their tangents -----------
  const double* x = tan ? dir_of(cd) : eval_pops(cd, mode);
  const double* Jd = jdag_ptr(cd);
  for (int i = threadIdx.x; i < nray * nz; i += blockDim.x) {
    const int y = i / nz, k = i - y * nz, yr = y >= R5 ? y - R5 : y, m = yr / Qb, ql = yr - m * Qb;
    if (ql >= nqb) continue;
    const int d = y >= R5 ? m : nmu + m, q = qb0 + ql;
    const size_t o = (size_t)d * per + (size_t)q * nz + k;
    const double* Vk = Vd + (size_t)d * dstride + k;
    const double* xk = x + (size_t)k * nl;
    const int* L = s_list + ql * kMaxT;
    double a = 0.0, e = 0.0;   // sum V (x_lo - g x_up), sum g V x_up
    for (int j = 0; j < kMaxT; ++j) {
      const int w = L[j];
      if (w < 0) break;
      const size_t p = (size_t)(w >> 8) * nz;
      const double V = Vk[p], gx = T.G[p + k] * xk[w & 15];
      a = fma(V, xk[(w >> 4) & 15] - gx, a);
      e = fma(V, gx, e);
    }
    const double c2 = T.c2[q];
    if (tan) {
      s0[k * rp + y] = a;
      s1[k * rp + y] = fma(c2, e, -cd.w.mS[o] * a) * cd.w.mchi[o];   // mchi: 1/chi
    } else {
      const size_t qk = (size_t)q * nz + k;
      const double sca = T.chi_sca[k], chi = T.chi_c[qk] + sca + a;
      const double eta = fma(c2, e, T.eta_c[qk] + sca * Jd[qk]);
      const double rc = 1.0 / chi, s = eta * rc, S = fma(fma(-s, chi, eta), rc, s);   // rounded once
      s0[k * rp + y] = chi;
      s1[k * rp + y] = S;
      if (base) {
        cd.w.mchi[o] = rc;
        cd.w.mS[o] = S;
      }
    }
  }
  __syncthreads();
  if (!tan) {
    for (int i = threadIdx.x; i < nray * (nz - 1); i += blockDim.x) {
      const int l = i / nray, y = i - l * nray, yr = y >= R5 ? y - R5 : y, m = yr / Qb;
      if (yr - m * Qb >= nqb) continue;
      const double dtau = T.dz[l] * s_inv2mu[m] * (s0[l * rp + y] + s0[(l + 1) * rp + y]), hw = s_hw[m];
      double e, w, a, bq, om;
      step_coef(dtau, 1.0 / dtau, s_tab, e, w, a, bq, om);
      double* p = cf + (size_t)l * kMvPlanes * nray + y;
      p[0] = e;
      p[nray] = hw * a;
      p[2 * nray] = hw * (bq * dtau);
      p[3 * nray] = hw * bq;
    }
    __syncthreads();
    load(0);
  }
  // ---- recurrences: h I^k = h I^u e + X ----------------------------------------
  double I = 0.0;   // boundary values (their tangents are zero)
  if (run) {
    if (up && !tan) I = s_hw[rm] * T.Bn[(size_t)(qb0 + rq) * nz + nz - 1];
    sI[(up ? nz - 1 : 0) * rp + ray] = I;
  }
  store(0);
  load(1);
  __syncthreads();
  for (int c = 0; c < nch; ++c) {
    if (!helper) {
      if (run) {
        const int c0 = c * kChunk, rows = min(kChunk, nz - 1 - c0);
        const double* in = s_in + (size_t)(c & 1) * 2 * kChunk * nray + ray;
        double e[kChunk], X[kChunk];
#pragma unroll
        for (int r = 0; r < kChunk; ++r) {
          const int q = min(r, rows - 1) * nray;
          e[r] = in[q];
          X[r] = in[kChunk * nray + q];
        }
#pragma unroll
        for (int r = 0; r < kChunk; ++r) X[r] = I = r < rows ? fma(I, e[r], X[r]) : I;
#pragma unroll
        for (int r = 0; r < kChunk; ++r)
          if (r < rows) sI[(up ? nz - 2 - c0 - r : c0 + r + 1) * rp + ray] = X[r];
      }
    } else if (c + 1 < nch) {
      store(c + 1);
      load(c + 2);
    }
    __syncthreads();
  }
  if (base) {
    if (run && up) cd.w.Iem[(size_t)(qb0 + rq) * nmu + rm] = I / s_hw[rm];
    // the slope of each ray's intensity on its optical depth, times h |dz|/(2 mu)
    for (int i = threadIdx.x; i < nray * (nz - 1); i += blockDim.x) {
      const int l = i / nray, y = i - l * nray, yr = y >= R5 ? y - R5 : y, m = yr / Qb;
      if (yr - m * Qb >= nqb) continue;
      const bool u = y >= R5;
      const int k = u ? l : l + 1, ku = u ? l + 1 : l;
      double* p = cf + (size_t)l * kMvPlanes * nray + y;
      const double Su = s1[ku * rp + y], e = p[0];
      const double G = fma(p[3 * nray], s1[k * rp + y] - Su, e * fma(s_hw[m], Su, -sI[ku * rp + y]));
      const double hG = T.dz[l] * s_inv2mu[m] * G;
      p[3 * nray] = hG;
      s0[k * rp + y] = hG;   // chi is no longer needed; the boundary depth is set below
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nray * nz; i += blockDim.x) {
      const int y = i / nz, k = i - y * nz, yr = y >= R5 ? y - R5 : y, m = yr / Qb, ql = yr - m * Qb;
      if (ql >= nqb) continue;
      const bool u = y >= R5;
      const int l = u ? k : k - 1, e = k * rp + y;
      double lx = 0.0, le = 0.0;
      if (l >= 0 && l < nz - 1) {
        const size_t o = (size_t)(u ? m : nmu + m) * per + (size_t)(qb0 + ql) * nz + k;
        le = cd.w.mchi[o] * cf[((size_t)l * kMvPlanes + 1) * nray + y];
        lx = fma(-s1[e], le, s0[e]);
      }
      s0[e] = lx;   // h dI/dchi, h dI/deta
      s1[e] = le;
    }
    __syncthreads();
    // J = sum of h I over the rays
    for (int i = threadIdx.x; i < nqb * nz; i += blockDim.x) {
      const int ql = i / nz, k = i - ql * nz;
      double J = 0.0;
      for (int m = 0; m < 2 * nmu; ++m) J += sI[k * rp + m * Qb + ql];
      jnew_ptr(cd)[(size_t)(qb0 + ql) * nz + k] = J;
    }
  }
  // ---- parts of the rate integrals (and of the block-Jacobi sums) -------------
  for (int i = threadIdx.x; i < s_nact * nz; i += blockDim.x) {
    const int a = i / nz, k = i - a * nz, t = s_act[a];
    const int q0 = T.t_q0[t], qa = max(q0, qb0), qe = min(T.t_q1[t], qb0 + nqb - 1);
    const double nlo = x[k * nl + T.t_lo[t]], nup = x[k * nl + T.t_up[t]];
    double a0 = 0.0, a1 = 0.0;
    double acc[kMaxL];
    if (base)
      for (int j = 0; j < nl; ++j) acc[j] = 0.0;
    for (int q = qa; q <= qe; ++q) {
      const int p = T.t_base[t] + q - q0, ql = q - qb0;
      const size_t pk = (size_t)p * nz + k;
      const double W = T.t_w[p] * T.rw[q], gt = T.G[pk], c2 = T.c2[q];
      double V[2 * kMaxMu], su = 0.0, sv = 0.0;
#pragma unroll
      for (int m = 0; m < 2 * nmu; ++m)   // ray order: ingoing, then outgoing
        V[m] = Vd[(size_t)(m < nmu ? nmu + m : m - nmu) * dstride + pk];
#pragma unroll
      for (int m = 0; m < 2 * nmu; ++m) {
        su = fma(V[m], sI[k * rp + m * Qb + ql], su);
        if (!tan) sv = fma(s_hw[m < nmu ? m : m - nmu], V[m], sv);
      }
      a0 = fma(W, su, a0);
      a1 = fma(W * gt, tan ? su : fma(c2, sv, su), a1);
      if (base) {
        const double c = W * fma(-gt, nup, nlo);
        const int* L = s_list + ql * kMaxT;
        for (int j = 0; j < kMaxT; ++j) {
          const int w = L[j];
          if (w < 0) break;
          const size_t ps = (size_t)(w >> 8) * nz + k;
          double m1 = 0.0, m2 = 0.0;
#pragma unroll
          for (int m = 0; m < 2 * nmu; ++m) {
            const double vv = V[m] * Vd[(size_t)(m < nmu ? nmu + m : m - nmu) * dstride + ps];
            m1 = fma(vv, s0[k * rp + m * Qb + ql], m1);
            m2 = fma(vv, s1[k * rp + m * Qb + ql], m2);
          }
          acc[(w >> 4) & 15] = fma(c, m1, acc[(w >> 4) & 15]);
          acc[w & 15] = fma(c * T.G[ps], fma(c2, m2, -m1), acc[w & 15]);
        }
      }
    }
    double* part = cd.w.rpart + (size_t)s_off[a] * nslot * nz + k;
    part[0] = a0;
    part[nz] = a1;
    if (base)
      for (int j = 0; j < nl; ++j) part[(size_t)(2 + j) * nz] = acc[j];
  }
}

int launch_eval64_moving(const Batch& b, cudaStream_t s) {
  const dim3 g(b.max_tiles, b.ncols);
  if (b.eval_mu == 5) k_eval64_moving<5><<<g, kEvalThreads, b.eval_smem, s>>>(b.d_cols);
  else k_eval64_moving<0><<<g, kEvalThreads, b.eval_smem, s>>>(b.d_cols);
  JFNK_CUDA(cudaGetLastError());
  return JFNK_OK;
}

int cached_prepare() {
  ExpEntry tab[kExpTab];
  for (int j = 0; j < kExpTab; ++j) tab[j] = exp_entry(j);
  JFNK_CUDA(cudaMemcpyToSymbol(d_exp_tab, tab, sizeof(tab)));
  JFNK_CUDA(cudaFuncSetAttribute(k_eval64<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCachedSmem));
  JFNK_CUDA(cudaFuncSetAttribute(k_eval64<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCachedSmem));
  JFNK_CUDA(cudaFuncSetAttribute(k_eval64_moving<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCachedSmem));
  JFNK_CUDA(cudaFuncSetAttribute(k_eval64_moving<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCachedSmem));
  return JFNK_OK;
}

// Five angles (every workload's count) have an instantiation; the others run the
// loops over them at run time and lie on the same line: a residual of 82 depths x
// 1,005 frequencies takes 94, 98, 103, 112 us with 1 to 4 angles, 123 with 5, 131, 144
// and 153 with 6 to 8.
int launch_eval64(const Batch& b, cudaStream_t s) {
  const dim3 g(b.max_tiles, b.ncols);
  if (b.eval_mu == 5) k_eval64<5><<<g, kEvalThreads, b.eval_smem, s>>>(b.d_cols, b.d_opts);
  else k_eval64<0><<<g, kEvalThreads, b.eval_smem, s>>>(b.d_cols, b.d_opts);
  JFNK_CUDA(cudaGetLastError());
  return JFNK_OK;
}

}  // namespace jfnk
