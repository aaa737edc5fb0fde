// The weighting function s(r) of the environment matrix (Sec. II) and its derivative, shared by
// env_force.cu's kernels and the tensor-core tabulation's fused rows (tabulate_tc.cu), so that both form
// the same bits.  P supplies rcs, rc, inv_width = 1 / (rc - rcs) and kind; real is double, float or
// df64.
#pragma once

#include "dp_common.cuh"
#include "fixed.cuh"

namespace dpc {
namespace {

__device__ __forceinline__ double recip(const double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(const float x) { return 1.0f / x; }
__device__ __forceinline__ df64 recip(const df64 x) { return dfl::rcp(x); }
__device__ __forceinline__ void sin_cos_pi(const double u, double *s, double *c) { sincospi(u, s, c); }
__device__ __forceinline__ void sin_cos_pi(const float u, float *s, float *c) { sincospif(u, s, c); }
__device__ __forceinline__ void sin_cos_pi(const df64 u, df64 *s, df64 *c) { dfl::sincospi(u, s, c); }
template <typename real>
__device__ __forceinline__ real half_pi() { return real(1.57079632679489661923); }
template <>
__device__ __forceinline__ df64 half_pi<df64>() { return df64(1.5707964e+00f, -4.371139e-08f); }

// s(r) and ds/dr of the weighting function (Sec. II).  u = (r - rcs)/(rc - rcs);
// kind 1: w = u^3 (-6u^2 + 15u - 10) + 1 (the paper's switch), w' = -30 u^2 (u - 1)^2;
// kind 0: w = cos(pi u)/2 + 1/2, w' = -(pi/2) sin(pi u).  inv_r = 1/r.
template <typename real, typename EP>
__device__ __forceinline__ void weight(const EP &P, real r, real inv_r, real &sv, real &dsv) {
  if (r < P.rcs) {
    sv = inv_r;
    dsv = -inv_r * inv_r;
  } else if (r < P.rc) {
    const real u = (r - P.rcs) * P.inv_width;
    real w, dw;
    if (P.kind == 1) {
      const real u2 = u * u, um = u - real(1);
      w = fma(u2 * u, fma(fma(real(-6), u, real(15)), u, real(-10)), real(1));
      dw = real(-30) * u2 * um * um;
    } else {
      real sn, cs;
      sin_cos_pi(u, &sn, &cs);
      w = fma(real(0.5), cs, real(0.5));
      dw = -(half_pi<real>() * sn);
    }
    sv = w * inv_r;
    dsv = (dw * P.inv_width - w * inv_r) * inv_r;
  } else {
    sv = real(0);
    dsv = real(0);
  }
}

// r = sqrt(r2) and 1/r.
template <typename real>
__device__ __forceinline__ void radius(real r2, real &r, real &inv_r) {
  r = sqrt(r2);
  inv_r = recip(r);
}
// In f64: from the float 1/sqrt (its argument's and result's fields moved by integer operations) by one step of
// third order, y (1 + e/2 + 3 e^2/8) with e = 1 - r2 y^2 below 2^-20, and r = r2 y with its own residual taken off
// (r2 - r^2) y / 2: eight FP64 instructions where the square root and the division took about twenty.  1/r within a
// unit of the last place, r rounded as by sqrt but for near ties; without the residual r was off by up to 1.6 units,
// which in the switch's tail made ds/dr 1.5 times less exact.
__device__ __forceinline__ void radius(double r2, double &r, double &inv_r) {
  const unsigned hi = (unsigned)__double2hiint(r2), lo = (unsigned)__double2loint(r2);
  if (hi - 0x39b00000u >= 0x0c800000u) {  // outside [2^-100, 2^100), negative, NaN
    r = sqrt(r2);
    inv_r = 1.0 / r;
    return;
  }
  const unsigned y = __float_as_uint(rsqrtf(__uint_as_float((hi - 0x38000000u) << 3 | lo >> 29)));
  const double y0 = __hiloint2double((int)((y >> 3) + 0x38000000u), (int)(y << 29));
  const double e = fma(-(r2 * y0), y0, 1.0);
  inv_r = fma(y0, fma(0.375, e, 0.5) * e, y0);
  r = r2 * inv_r;
  r = fma(fma(-r, r, r2), __hiloint2double(__double2hiint(inv_r) - (1 << 20), __double2loint(inv_r)), r);
}

// weight() in f64: the switch and its derivative are polynomials of u in fixed point (fixed.cuh; units of
// 2^-60 or 2^-58), with no FP64 instruction but the conversions of u and of the results:
//   kind 1: w = 1 + 8 u^3 ((-6 u^2 + 15 u - 10) / 8), w' = -30 (u (u - 1))^2;
//   kind 0: with x = u - 1/2, z = x^2 <= 1/4, cos(pi u) = -sin(pi x) and sin(pi u) = cos(pi x) by their Taylor
//           series in z, twelve terms each (the next is below 2^-63), coefficients over 4.
// Why: a row's environment took 50 (kind 1) to 66 (kind 0) FP64 instructions, 68 clocks of a sub-partition
// each, and set the time of the kernels that form rows; now it takes 25.  Measured (copper, 4,096 atoms, kind 1):
// the fused forward's runs kernel 0.196 -> 0.160 ms, the fused rows and forces 0.345 -> 0.312 ms; water (1,536
// atoms, kind 0) 0.039 -> 0.030 and 0.051 -> 0.036 ms.  w and w' have absolute errors; near the cut-off, where both
// are small, s and ds/dr are still more exact than with w from FP64, whose cancellation there is the larger error.
struct SwitchFixed {
  long long w, dw;  // units of 2^-60 and 2^-58
};
__device__ __forceinline__ SwitchFixed switch_fixed(int kind, long long u) {
  constexpr int L = 30;
  using fx::Fix;
  SwitchFixed S;
  if (kind == 1) {  // uniform
    const Fix uf = fx::limbs<L>(u);
    const long long u2 = fx::mul<L>(uf, uf);
    const long long u3 = fx::mul<L>(fx::limbs<L>(u2), uf);
    const long long q8 = (2 * u - (u >> 3)) - (u2 - (u2 >> 2)) - (5ll << 58);
    S.w = (1ll << 60) + 8 * fx::mul<L>(fx::limbs<L>(u3), fx::limbs<L>(q8));
    const Fix uv = fx::limbs<L>(u2 - u);  // u (u - 1)
    S.dw = -(15 * fx::mul<L>(uv, uv) >> 1);
  } else {
    constexpr long long kSin[12] = {905502432259640355, -1489491798437810879, 735034740462416105, -172726240700510392,
                                    23676939797241351,  -2124382083883464,    134402633106998,    -6316670567766,
                                    229202351602,       -6614434322,          155432976,          -3031743};
    constexpr long long kCos[12] = {452751216129820178, -2234237697656716318, 1837586851156040263, -604541842451786371,
                                    106546229087586079, -11684101461359051,   873617115195484,     -47375029258244,
                                    1948219988620,      -62837126059,         1632046252,          -34865045};
    const Fix x = fx::limbs<L>(u - (1ll << 59));
    const Fix z = fx::limbs<L>(fx::mul<L>(x, x));
    long long p = kSin[11], q = kCos[11];
#pragma unroll
    for (int k = 10; k >= 0; --k) {
      p = kSin[k] + fx::mul<L>(fx::limbs<L>(p), z);
      q = kCos[k] + fx::mul<L>(fx::limbs<L>(q), z);
    }
    S.w = (1ll << 59) - 2 * fx::mul<L>(fx::limbs<L>(p), x);  // p: sin(pi x) / (4 x)
    S.dw = -q;                                              // q: (pi / 2) cos(pi x) / 4
  }
  return S;
}
template <typename EP>
__device__ __forceinline__ void weight(const EP &P, double r, double inv_r, double &sv, double &dsv) {
  // r >= 0, compared as integers: a NaN's bits, its sign off, lie above every radius.  (The bits through PTX: of a
  // square root the compiler takes the sign to be off already, which is not so for a NaN.)
  long long rb;
  asm("mov.b64 %0, %1;" : "=l"(rb) : "d"(r));
  rb &= 0x7fffffffffffffffll;
  if (rb < __double_as_longlong(P.rcs)) {
    sv = inv_r;
    dsv = -inv_r * inv_r;
  } else if (rb < __double_as_longlong(P.rc)) {
    const SwitchFixed S = switch_fixed(P.kind, fx::from_double((r - P.rcs) * P.inv_width, 60));
    // (rounded by itself: no kernel may fuse it into what it does next, or their rows would not be the same bits)
    sv = __dmul_rn(fx::to_double(S.w, -60), inv_r);
    dsv = fma(fx::to_double(S.dw, -58), P.inv_width, -sv) * inv_r;
  } else {
    sv = 0.0;
    dsv = 0.0;
  }
}

// The environment's parameters checked on the host (DP_ERR_NULL / DP_ERR_TABLE_INFO).
inline int check_env(const dp_env_info *env) {
  if (!env) return set_error(DP_ERR_NULL, "env is NULL");
  if (!(env->rcs > 0.0) || !(env->rc > env->rcs))
    return set_error(DP_ERR_TABLE_INFO, "need 0 < rcs < rc (rcs %g, rc %g)", env->rcs, env->rc);
  if (env->kind != 0 && env->kind != 1) return set_error(DP_ERR_TABLE_INFO, "switch kind %d not 0 or 1", env->kind);
  if (!(env->std > 0.0) || !(env->std_all > 0.0))
    return set_error(DP_ERR_TABLE_INFO, "normalisation needs std > 0 and std_all > 0");
  if (!isfinite(env->mean)) return set_error(DP_ERR_TABLE_INFO, "normalisation mean not finite");
  return DP_OK;
}

}  // namespace
}  // namespace dpc
