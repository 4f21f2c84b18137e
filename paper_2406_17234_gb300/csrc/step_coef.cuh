// FP64 coefficients of one step of the formal solution (App. A.1) for the
// cached evaluation. Plain C++ outside nvcc, so that their accuracy can be
// measured on the host against multi-precision values.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define JFNK_HD __host__ __device__ __forceinline__
#else
#define JFNK_HD inline
#endif

namespace jfnk {

constexpr int kExpTab = 256;
struct alignas(16) ExpEntry {
  double p, q;   // 2^(-j/256) and 1 - 2^(-j/256)
};
inline ExpEntry exp_entry(int j) {
  return {std::exp2(-j / (double)kExpTab), -std::expm1(-j / (double)kExpTab * 0.69314718055994530942)};
}

JFNK_HD int hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
JFNK_HD int lo_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2loint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (int)(uint32_t)b;
#endif
}
JFNK_HD double from_words(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const uint64_t b = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

// e = e^(-x) and om = 1 - e for x >= 1e-3 (e = 0 from x = 700 on) in eleven FP64
// instructions: x = n ln2/256 + r, |r| < 1.4e-3, 2^(-n/256) from a table, p =
// e^(-r) - 1 to the fifth order (the next term is below 1e-20): the table
// method of Tang (ACM Trans. Math. Softw. 15, 144, 1989). Below ln 2 the sum is
// formed for om, from tabulated 1 - 2^(-j/256), and e = 1 - om: om then keeps
// its relative accuracy (2e-16) in thin layers, where 1 - e cancels.
JFNK_HD void neg_exp(double x, const ExpEntry* tab, double& e, double& om) {
  const double magic = 6755399441055744.0;   // 1.5 2^52: n in the low word
  const double t = fma(x, 369.32993046757464, magic);
  const int n = lo_word(t);
  const double tn = t - magic;
  double r = fma(tn, -0.0027076061740622863, x);
  r = fma(tn, -9.0587766165870294e-20, r);
  double q = fma(r, -1.0 / 120, 1.0 / 24);
  q = fma(q, r, -1.0 / 6);
  q = fma(q, r, 0.5);
  q = fma(q, r, -1.0);
  const ExpEntry T0 = tab[n & (kExpTab - 1)];
  const double T = from_words(hi_word(T0.p) - ((n >> 8) << 20), lo_word(T0.p));
  const bool small = n < kExpTab;
  const double u = fma(small ? -T : T, q * r, small ? T0.q : T), v = 1.0 - u;
  e = small ? v : u;
  om = small ? u : v;
  if (hi_word(x) >= 0x4085e000) {   // x >= 700
    e = 0.0;
    om = 1.0;
  }
}

// Coefficients of one step of optical depth x, r = 1/x (App. A.1): e = exp(-x),
// w = (1 - e)/x, bq = (w - e)/x, a = 1 - w and om = 1 - e = a + bq x. The direct
// forms lose 2e-16/x relative in a and bq (4e-13 at x = 1e-3), so below 1e-3
// the Taylor series w = sum (-x)^n/(n+1)!, a/x = sum (-x)^n/(n+2)! and bq =
// sum (-x)^n (n+1)/(n+2)! take over, to n = 4 (the next terms are below 2e-18
// there); they skip the exponential. (With the series from 1e-5 down only, a
// and bq lost up to 4e-11 in between.)
JFNK_HD void step_coef(double x, double r, const ExpEntry* tab, double& e, double& w, double& a, double& bq,
                       double& om) {
  if (x < 1e-3) {
    if (x > -1e-3) {
      w = fma(fma(fma(fma(1.0 / 120, x, -1.0 / 24), x, 1.0 / 6), x, -0.5), x, 1.0);
      bq = fma(fma(fma(fma(1.0 / 144, x, -1.0 / 30), x, 1.0 / 8), x, -1.0 / 3), x, 0.5);
      a = x * fma(fma(fma(fma(1.0 / 720, x, -1.0 / 120), x, 1.0 / 24), x, -1.0 / 6), x, 0.5);
      om = x * w;
      e = 1.0 - om;
      return;
    }
    om = -expm1(-x);   // inverted populations: x < 0
    e = 1.0 - om;
  } else {
    neg_exp(x, tab, e, om);
  }
  w = om * r;
  a = 1.0 - w;
  bq = (w - e) * r;
}

}  // namespace jfnk
