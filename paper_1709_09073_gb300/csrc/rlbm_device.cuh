// Device arithmetic of the fused stream-collide update (FP64 form).
//
// Per cell: moments N^mu, T^{mu nu} (Eqs. 20, 22) -> Landau frame (Eq. 21) ->
// n, theta, z (Eqs. 23-25) -> the 36 equilibrium moments in harmonic form
// (Appendix) -> the fifth-order discrete equilibrium as a block-diagonal
// projection (Eqs. 10-11) -> Anderson-Witting relaxation (Eq. 3).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rlbm_common.h"
#include "rlbm_tables.h"

namespace rlbm {

// ---------------------------------------------------------------- tables
// Each translation unit that includes this header gets its own copy.
static __constant__ double c_p[3][6] = {RLBM_P_MJ_INIT, RLBM_P_FD_INIT, RLBM_P_BE_INIT};
static __constant__ double c_w[3][6] = {RLBM_W_MJ_INIT, RLBM_W_FD_INIT, RLBM_W_BE_INIT};
static __constant__ double c_p2[3][6] = {RLBM_P2_MJ_INIT, RLBM_P2_FD_INIT, RLBM_P2_BE_INIT};
// projection tables per expansion order N = 2..5 (index N - 2; entries of degree
// above N are zero) and EDF
static __constant__ double c_Q[4][3][126] = {
    {RLBM_QO2_MJ_INIT, RLBM_QO2_FD_INIT, RLBM_QO2_BE_INIT},
    {RLBM_QO3_MJ_INIT, RLBM_QO3_FD_INIT, RLBM_QO3_BE_INIT},
    {RLBM_QO4_MJ_INIT, RLBM_QO4_FD_INIT, RLBM_QO4_BE_INIT},
    {RLBM_Q_MJ_INIT, RLBM_Q_FD_INIT, RLBM_Q_BE_INIT}};
// exact defects of the rounded Q tables in the conserved moments: e1 (N^0, block
// k = 0), e2 (T^00, block 0), e3 (T^0x + i T^0y, block 1), 6 entries each
static __constant__ double c_E[4][3][18] = {
    {RLBM_EO2_MJ_INIT, RLBM_EO2_FD_INIT, RLBM_EO2_BE_INIT},
    {RLBM_EO3_MJ_INIT, RLBM_EO3_FD_INIT, RLBM_EO3_BE_INIT},
    {RLBM_EO4_MJ_INIT, RLBM_EO4_FD_INIT, RLBM_EO4_BE_INIT},
    {RLBM_E_MJ_INIT, RLBM_E_FD_INIT, RLBM_E_BE_INIT}};
constexpr int kOrder5 = 3;  // table index of the fifth order
// FP32 tables, rounded at compile time (a conversion in the kernel would take the FP64
// unit): the same defects, for the correction itself (see eq_moments), the series of g_2
// and g_3 in t, and the reversion t(w)
struct TablesF {
  float e[4][3][18], logser[2][12], rev[RLBM_NREV];
};
constexpr TablesF make_tables_f() {
  constexpr double e[4][3][18] = {{RLBM_EO2_MJ_INIT, RLBM_EO2_FD_INIT, RLBM_EO2_BE_INIT},
                                  {RLBM_EO3_MJ_INIT, RLBM_EO3_FD_INIT, RLBM_EO3_BE_INIT},
                                  {RLBM_EO4_MJ_INIT, RLBM_EO4_FD_INIT, RLBM_EO4_BE_INIT},
                                  {RLBM_E_MJ_INIT, RLBM_E_FD_INIT, RLBM_E_BE_INIT}};
  constexpr double ls[5 * RLBM_NLOGSER] = RLBM_LOGSER_INIT;
  constexpr double rv[RLBM_NREV] = RLBM_REV_INIT;
  TablesF t{};
  for (int i = 0; i < 12; ++i) {
    t.logser[0][i] = (float)ls[i];
    t.logser[1][i] = (float)ls[RLBM_NLOGSER + i];
  }
  for (int i = 0; i < RLBM_NREV; ++i) t.rev[i] = (float)rv[i];
  for (int o = 0; o < 4; ++o)
    for (int d = 0; d < 3; ++d)
      for (int i = 0; i < 18; ++i) t.e[o][d][i] = (float)e[o][d][i];
  return t;
}
static __constant__ TablesF c_tf = make_tables_f();
static __constant__ double c_pnk[63] = RLBM_PNK_INIT;
static __constant__ double c_logser[5 * RLBM_NLOGSER] = RLBM_LOGSER_INIT;
static __constant__ double c_invpow[6 * RLBM_NSERIES] = RLBM_INVPOW_INIT;
static __constant__ double c_be_exp[6 * RLBM_NEXP] = RLBM_BE_EXP_INIT;
static __constant__ double c_fd_exp[6 * RLBM_NEXP] = RLBM_FD_EXP_INIT;
static __constant__ double c_be_logcoef[6] = RLBM_BE_LOGCOEF_INIT;
static __constant__ double c_be_harm[6] = RLBM_BE_HARM_INIT;
static __constant__ double c_g_zc[6] = RLBM_G_ZC_INIT;

// Offset of harmonic block k in the Q tables: sum_{k'<k} 6 (6 - k').
__host__ __device__ constexpr int qoff(int k) { return 6 * (6 * k - (k * (k - 1)) / 2); }

// Moment polynomials P_nk(u^2) (Appendix), entry 3 * (n(n+1)/2 + k) + power: a
// compile-time function, so that the 42 coefficients that are 0 cost nothing.
__host__ __device__ constexpr double pnk(int i) {
  constexpr double t[63] = RLBM_PNK_INIT;
  return t[i];
}

// ------------------------------------- FP32 <-> FP64 on the integer pipe
// The conversion instructions run on the FP64 unit too. Where an FP32 value only starts
// or scales an FP64 correction, the bits are moved by integer instructions instead.
// double -> float, cut towards zero; below the normal range 0, above it (and for
// infinity and NaN) infinity
__device__ __forceinline__ float cut_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), m = hi & 0x7fffffffu;
  unsigned t = ((m - 0x38000000u) << 3) | (lo >> 29);
  if (m < 0x38100000u) t = 0u;
  if (m >= 0x47f00000u) t = 0x7f800000u;
  return __uint_as_float(t | (hi & 0x80000000u));
}
// float -> double, exact for normal values and zeros; denormals go to 0. (Infinity and
// NaN give a finite value: the caller's own test sends those states elsewhere.)
__device__ __forceinline__ double widen_f64(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  return m < 0x00800000u ? __hiloint2double((int)(b & 0x80000000u), 0)
                         : __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}

// ------------------------------------------------ FP64 divide and square root
// GB300 issues one FP64 warp instruction per SM sub-partition every 64 clocks, so a
// reciprocal or a root costs what its FP64 instructions cost. Both start from the
// FP32 unit's value r (about 23 bits) and take three terms of a series in FP64: with
// e = 1 - x r, 1/x = r (1 + e + e^2 + ...), and with e = 1 - x r^2, 1/sqrt(x) =
// r (1 + e/2 + 3 e^2/8 + ...); the terms left out are below 2^-64. Largest relative
// errors: rcp64 half an ulp, as the division; rsqrt64 1.5 * 2^-53, where 1 / sqrt(x)
// rounds twice. Outside the FP32 range they fall back to the compiler's own. (A quotient
// a * rcp64(b) rounds once more than a / b. With the residual applied, as the division
// has it, the read-out temperature's error is the same to 1 % and the FP64 steps take
// 0.4 % longer: not taken.)
__device__ __forceinline__ double rcp64(double x) {
  const float xf = cut_f32(x);
  if (!(fabsf(xf) > 1e-30f && fabsf(xf) < 1e30f)) return 1.0 / x;
  const double r = widen_f64(1.0f / xf);
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rsqrt64(double x) {
  const float xf = cut_f32(x);
  if (!(xf > 1e-30f && xf < 1e30f)) return 1.0 / sqrt(x);
  const double r = widen_f64(rsqrtf(xf));
  const double e = fma(-(x * r), r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

// ------------------------------------------------------- EDF integrals g_nu
// g[nu-1] = g_nu(z), nu = 1..6 (Eq. 12). MJ: z. BE: Li_nu(z). FD: -Li_nu(-z).
// Power series in z for small z, the expansions in mu = ln z around z = 1
// (zeta values for BE, eta values for FD), and for FD z > 4 the inversion
// formula -Li_nu(-z) = (-1)^nu Li_nu(-1/z) + (ln z)^nu/nu! + 2 sum_j eta(2j) (ln z)^{nu-2j}/(nu-2j)!.
__device__ __forceinline__ void li_series6(double x, double g[6]) {
  // sum_{k>=1} x^k k^{-nu}, |x| <= 1/4
  double xk = 1.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) g[i] = 0.0;
  for (int k = 1; k <= RLBM_NSERIES; ++k) {
    xk *= x;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = fma(xk, c_invpow[i * RLBM_NSERIES + k - 1], g[i]);
    if (fabs(xk) < 1e-18) break;
  }
}

template <int EDF>
__device__ void g_all(double z, double g[6]) {
  if (EDF == EDF_MJ) {
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = z;
    return;
  }
  if (EDF == EDF_BE) {
    if (z <= 0.25) { li_series6(z, g); return; }
    const double mu = log(z);
    double mk = 1.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = 0.0;
    for (int k = 0; k < RLBM_NEXP; ++k) {
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = fma(mk, c_be_exp[i * RLBM_NEXP + k], g[i]);
      mk *= mu;
      if (fabs(mk) < 1e-30) break;
    }
    // the k = nu-1 term: mu^{nu-1}/(nu-1)! (H_{nu-1} - ln(-mu))
    const double lnm = log(-mu);
    double mp = 1.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      g[i] = fma(mp * c_be_logcoef[i], c_be_harm[i] / c_be_logcoef[i] - lnm, g[i]);
      mp *= mu;
    }
    return;
  }
  // FD
  if (z <= 0.25) {
    li_series6(-z, g);
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = -g[i];
    return;
  }
  if (z <= 4.0) {
    const double mu = log(z);
    double mk = 1.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = 0.0;
    for (int k = 0; k < RLBM_NEXP; ++k) {
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = fma(mk, c_fd_exp[i * RLBM_NEXP + k], g[i]);
      mk *= mu;
      if (fabs(mk) < 1e-30) break;
    }
    return;
  }
  li_series6(-1.0 / z, g);
  const double L = log(z);
  // eta(2) = pi^2/12, eta(4) = 7 pi^4/720, eta(6) = 31 pi^6/30240
  const double eta2 = 0.82246703342411321824, eta4 = 0.94703282949724591758,
               eta6 = 0.98555109129743510410;
  const double L2 = L * L, L3 = L2 * L, L4 = L3 * L, L5 = L4 * L, L6 = L5 * L;
  g[0] = -g[0] + L;
  g[1] = g[1] + L2 / 2.0 + 2.0 * eta2;
  g[2] = -g[2] + L3 / 6.0 + 2.0 * eta2 * L;
  g[3] = g[3] + L4 / 24.0 + 2.0 * eta2 * L2 / 2.0 + 2.0 * eta4;
  g[4] = -g[4] + L5 / 120.0 + 2.0 * eta2 * L3 / 6.0 + 2.0 * eta4 * L;
  g[5] = g[5] + L6 / 720.0 + 2.0 * eta2 * L4 / 24.0 + 2.0 * eta4 * L2 / 2.0 + 2.0 * eta6;
}

// g_1, g_2, g_3 alone (g[0..2] of g_all): what the Newton iterations below need.
// In the series range g_1 has the closed form ln(1 + z) (FD) or -ln(1 - z) (BE),
// and g_2, g_3 take two series instead of six.
template <int EDF>
__device__ __forceinline__ void g123(double z, double g[3]) {
  if (EDF != EDF_MJ && z <= 0.25) {
    const double x = EDF == EDF_BE ? z : -z;
    double xk = 1.0, s2 = 0.0, s3 = 0.0;
    for (int k = 1; k <= RLBM_NSERIES; ++k) {
      xk *= x;
      s2 = fma(xk, c_invpow[RLBM_NSERIES + k - 1], s2);
      s3 = fma(xk, c_invpow[2 * RLBM_NSERIES + k - 1], s3);
      if (fabs(xk) < 1e-18) break;
    }
    g[0] = EDF == EDF_BE ? -log1p(-z) : log1p(z);
    g[1] = EDF == EDF_BE ? s2 : -s2;
    g[2] = EDF == EDF_BE ? s3 : -s3;
    return;
  }
  double g6[6];
  g_all<EDF>(z, g6);
  g[0] = g6[0];
  g[1] = g6[1];
  g[2] = g6[2];
}

// A Newton step d in mu leaves an error of about C d^2, C = |F''/(2F')| of the
// equation solved: at most 0.23 for FD and about 0.12/(1 - z) for BE (computed
// with arbitrary-precision polylogs for both solves below). A Newton step with
// d^2 C_bound < 1e-17 (C_bound = 0.25, or 0.25/(1 - z) for BE) is therefore
// accepted without evaluating the equation again.
template <int EDF>
__device__ __forceinline__ bool newton_done64(double d, double z) {
  const double cb = EDF == EDF_BE ? 0.25 / (1.0 - z) : 0.25;
  return d * d * cb < 1e-17;
}

// Fugacity from (eps, n), FD/BE: g_3^2/g_2^3 = (pi/2) eps^2/n^3 (Eq. 25), solved
// for mu = ln z by safeguarded Newton; BE states below R(z_c) are clamped.
// Start: with w = 1/target = g_2^3/g_3^2 = z + O(z^2), inverting the series gives
// mu = ln w - s w/2 + (119/1728) w^2 - s (85/6912) w^3 + O(w^4) (s = -1 FD, +1 BE),
// 1.4e-6 off in mu at z = 0.17: two Newton steps reach the FP64 floor, a third
// confirms it.
template <int EDF>
__device__ __noinline__ int solve_z_from_R_general(double target, double& z, double g[6]) {
  if (EDF == EDF_BE && target < RLBM_R_ZC) {
    z = ZC;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = c_g_zc[i];
    return ST_CLAMPED;
  }
  double lo = -60.0, hi = (EDF == EDF_BE) ? log(ZC) : 60.0;
  const double lt = log(target);
  double mu = -lt;
  const double w = 1.0 / target;
  if (w < 0.5) {
    constexpr double kS = EDF == EDF_BE ? 1.0 : -1.0;
    mu = fma(fma(fma(-kS * (85.0 / 6912.0), w, 119.0 / 1728.0), w, -0.5 * kS), w, mu);
  }
  mu = fmin(fmax(mu, lo + 1e-3), hi);
  int st = ST_ZSOLVE;
  double dprev = INFINITY;
  for (int it = 0; it < 80; ++it) {
    double gi[3];
    const double ze = exp(mu);
    g123<EDF>(ze, gi);
    const double F = log(gi[2] * gi[2] / (gi[1] * gi[1] * gi[1])) - lt;
    if (F == 0.0) { st = 0; break; }  // exact root at mu
    const double dF = 2.0 * gi[1] / gi[2] - 3.0 * gi[0] / gi[1];
    if (F > 0.0) lo = mu; else hi = mu;
    double mn = mu - F / dF;
    const bool newton = mn >= lo && mn <= hi;
    if (!newton) mn = 0.5 * (lo + hi);
    const double d = fabs(mn - mu);
    mu = mn;
    // converged: step at the tolerance, a Newton step whose error bound is below
    // it, or no longer shrinking at the noise floor
    if (d <= 1e-15 * fmax(1.0, fabs(mu)) || (newton && newton_done64<EDF>(d, ze)) ||
        (d < 1e-12 && d >= dprev)) {
      st = 0;
      break;
    }
    dprev = d;
  }
  z = exp(mu);
  g_all<EDF>(z, g);
  return st;
}

// Fugacity from (n, theta): n = 2 pi theta^2 g_2(z) (Eq. 25). Start: inverting
// G = g_2(z) gives mu = ln G +- G/4 - (5/288) G^2 +- G^3/288 + O(G^4) (upper
// signs FD, lower BE).
template <int EDF>
__device__ __noinline__ int solve_z_from_n_theta_general(double n, double theta, double& z, double g[6]) {
  const double G = n / (2.0 * PI * theta * theta);
  if (EDF == EDF_BE && G >= c_g_zc[1]) {
    z = ZC;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = c_g_zc[i];
    return ST_CLAMPED;
  }
  double lo = -60.0, hi = (EDF == EDF_BE) ? log(ZC) : 60.0;
  const double lG = log(G);
  double mu = lG;
  if (G < 0.5) {
    constexpr double kS = EDF == EDF_BE ? -1.0 : 1.0;
    mu = fma(fma(fma(kS / 288.0, G, -5.0 / 288.0), G, 0.25 * kS), G, mu);
  }
  mu = fmin(fmax(mu, lo + 1e-3), hi);
  int st = ST_ZSOLVE;
  double dprev = INFINITY;
  for (int it = 0; it < 80; ++it) {
    double gi[3];
    const double ze = exp(mu);
    g123<EDF>(ze, gi);
    const double F = log(gi[1]) - lG;      // increasing in mu
    if (F == 0.0) { st = 0; break; }       // exact root at mu
    const double dF = gi[0] / gi[1];
    if (F < 0.0) lo = mu; else hi = mu;
    double mn = mu - F / dF;
    const bool newton = mn >= lo && mn <= hi;
    if (!newton) mn = 0.5 * (lo + hi);
    const double d = fabs(mn - mu);
    mu = mn;
    // converged: step at the tolerance, a Newton step whose error bound is below
    // it, or no longer shrinking at the noise floor
    if (d <= 1e-15 * fmax(1.0, fabs(mu)) || (newton && newton_done64<EDF>(d, ze)) ||
        (d < 1e-12 && d >= dprev)) {
      st = 0;
      break;
    }
    dprev = d;
  }
  z = exp(mu);
  g_all<EDF>(z, g);
  return st;
}

// Fugacity in the variable t = g_1 = ln(1 + z) (FD) or -ln(1 - z) (BE), for t up
// to kTMax (z = 2.8 FD, 0.74 BE): there g_nu = t sum_n c_nu[n] (s t)^n (s = -1
// FD, +1 BE) with convergence radius 2 pi, so 11 to 28 terms of five series do what
// took 23 to 48 of six, and neither a logarithm nor an exponential is evaluated.
constexpr float kTMax = 1.35f;

// terms that put the first one left out below 2^-58 of the sum for every nu
__device__ __forceinline__ int logser_terms(float t) { return t <= 0.2f ? 12 : (t <= 0.45f ? 16 : (t <= 0.75f ? 20 : 28)); }

// g_2 and g_3 (FP32, 12 terms: 1e-7 at kTMax)
template <int EDF>
__device__ __forceinline__ void g23_t_f(float t, float& g2, float& g3) {
  const float u = EDF == EDF_BE ? t : -t, u2 = u * u;
  float a = 0.0f, b = 0.0f;
#pragma unroll
  for (int n = 10; n >= 2; n -= 2) a = fmaf(a, u2, c_tf.logser[0][n]);
#pragma unroll
  for (int n = 11; n >= 0; --n) b = fmaf(b, u, c_tf.logser[1][n]);
  g2 = t * fmaf(a, u2, fmaf(u, -0.25f, 1.0f));
  g3 = t * b;
}

// g_0 = z dg_1/dz (FP32): z/(1 + z) = 1 - e^-t (FD), z/(1 - z) = e^t - 1 (BE)
template <int EDF>
__device__ __forceinline__ float g0_t_f(float t) { return EDF == EDF_BE ? expm1f(t) : -expm1f(-t); }

// h_2 and h_3 of g_nu = t h_nu (even terms of h_2 beyond the second vanish, Li_2 - u +
// u^2/4 being odd)
template <int EDF>
__device__ __forceinline__ void h23_t(double t, int nt, double& h2, double& h3) {
  const double u = EDF == EDF_BE ? t : -t, u2 = u * u;
  double a = 0.0, b = 0.0;
  for (int n = nt; n >= 2; n -= 2) {
    a = fma(a, u2, c_logser[n]);
    b = fma(fma(b, u, c_logser[RLBM_NLOGSER + n + 1]), u, c_logser[RLBM_NLOGSER + n]);
  }
  h2 = fma(a, u2, fma(u, -0.25, 1.0));
  h3 = fma(fma(b, u, c_logser[RLBM_NLOGSER + 1]), u, c_logser[RLBM_NLOGSER]);
}

// h[nu - 1] of all six (h_1 = 1)
template <int EDF>
__device__ __forceinline__ void h_all_t(double t, int nt, double h[6]) {
  const double u = EDF == EDF_BE ? t : -t, u2 = u * u;
  double a = 0.0, b[4] = {0.0, 0.0, 0.0, 0.0};
  for (int n = nt; n >= 2; n -= 2) {
    a = fma(a, u2, c_logser[n]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      b[j] = fma(fma(b[j], u, c_logser[(j + 1) * RLBM_NLOGSER + n + 1]), u, c_logser[(j + 1) * RLBM_NLOGSER + n]);
  }
  h[0] = 1.0;
  h[1] = fma(a, u2, fma(u, -0.25, 1.0));
#pragma unroll
  for (int j = 0; j < 4; ++j)
    h[2 + j] = fma(fma(b[j], u, c_logser[(j + 1) * RLBM_NLOGSER + 1]), u, c_logser[(j + 1) * RLBM_NLOGSER]);
}

// z of t
template <int EDF>
__device__ __forceinline__ double z_of_t(double t) { return EDF == EDF_BE ? -expm1(-t) : expm1(t); }

// g_nu a step dmu of ln z (below 1e-9) beyond t: dg_nu/dmu = g_(nu-1), the second-order
// term is below 1e-18.
__device__ __forceinline__ void g_shift(double t, double dmu, float g0, const double h[6], double g[6]) {
#pragma unroll
  for (int i = 5; i >= 1; --i) g[i] = t * fma(dmu, h[i - 1], h[i]);
  g[0] = fma(dmu, widen_f64(g0), t);
}

// Fugacity from (eps, n), FD/BE: g_3^2/g_2^3 = target (Eq. 25). In t the ratio is
// w = 1/target = g_2^3/g_3^2 = t - (47/1728) t^3 - ..., so the reversion gives t to
// FP32 accuracy; one FP64 Newton step (in mu = ln z, whose F' = 2 g_2/g_3 - 3 g_1/g_2
// may be FP32) leaves about 1e-13, and the second one, taken from the residual at
// that point and carried to the six g_nu to first order, about 1e-20. Both residuals are
// formed with t divided out, from h_2, h_3 and w/t, all of order one: the squares of the
// g_nu leave the FP32 range below t = 1e-12, where a residual cut to zero would pass for
// a converged one. States outside the series' range, and any whose second step is not
// small, take the general solver. kZ: z is wanted (the step only needs the g_nu).
template <int EDF, bool kZ>
__device__ __forceinline__ int solve_z_from_R(double target, double& z, double g[6]) {
  const float wf = 1.0f / cut_f32(target);
  if (wf > 1e-20f && wf < 1.25f) {
    const float sw = EDF == EDF_BE ? wf : -wf;
    float p = 0.0f;
#pragma unroll
    for (int n = RLBM_NREV - 1; n >= 0; --n) p = fmaf(p, sw, c_tf.rev[n]);
    float tf = wf * p;
    if (wf > 0.5f) {  // the reversion's own series is short there: two FP32 steps
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        float a, b;
        g23_t_f<EDF>(tf, a, b);
        tf -= (a * a * a / (b * b) - wf) / fmaf(-47.0f / 576.0f, tf * tf, 1.0f);
      }
    }
    if (tf > 0.0f && tf <= kTMax) {
      const int nt = logser_terms(tf);
      double t = widen_f64(tf), h2, h3, h[6];
      h23_t<EDF>(t, nt, h2, h3);
      const float g0 = g0_t_f<EDF>(tf);
      {
        const double a = (target * t) * (h2 * h2 * h2);
        const float x = cut_f32(fma(h3, h3, -a)) / cut_f32(a), r2 = cut_f32(h2), r3 = cut_f32(h3);
        const float dmu = -x * fmaf(-0.5f, x, 1.0f) / (2.0f * r2 / r3 - 3.0f / r2);
        t += widen_f64(dmu * g0);
      }
      h_all_t<EDF>(t, nt, h);
      const double a = (target * t) * (h[1] * h[1] * h[1]);
      const float r2 = cut_f32(h[1]), r3 = cut_f32(h[2]);
      const float dmu = -(cut_f32(fma(h[2], h[2], -a)) / cut_f32(a)) / (2.0f * r2 / r3 - 3.0f / r2);
      if (fabsf(dmu) < 1e-9f) {
        g_shift(t, widen_f64(dmu), g0, h, g);
        if (kZ) z = z_of_t<EDF>(g[0]);
        return 0;
      }
    }
  }
  return solve_z_from_R_general<EDF>(target, z, g);
}

// Fugacity from (n, theta): n = 2 pi theta^2 g_2(z), as solve_z_from_R with
// G = g_2 = t + s t^2/4 + ... inverted in FP32 by Newton (dg_2/dt = t / g_0).
template <int EDF, bool kZ>
__device__ __forceinline__ int solve_z_from_n_theta(double n, double theta, double& z, double g[6]) {
  const double G = n / (2.0 * PI * theta * theta);
  if (EDF == EDF_MJ) {
    z = G;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = G;
    return 0;
  } else {
    const float Gf = cut_f32(G);
    if (Gf > 1e-20f && Gf < 1.25f) {
      float tf = Gf * fmaf(Gf, fmaf(7.0f / 72.0f, Gf, EDF == EDF_BE ? 0.25f : -0.25f), 1.0f);
      if (EDF == EDF_BE) tf = fminf(tf, kTMax);
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        float a, b;
        g23_t_f<EDF>(tf, a, b);
        tf -= (a - Gf) * g0_t_f<EDF>(tf) / tf;
      }
      if (tf > 0.0f && tf <= kTMax) {
        const int nt = logser_terms(tf);
        double t = widen_f64(tf), h2, h3, h[6];
        h23_t<EDF>(t, nt, h2, h3);
        const float g0 = g0_t_f<EDF>(tf);
        t += widen_f64(cut_f32(fma(-t, h2, G)) * g0 / tf);
        h_all_t<EDF>(t, nt, h);
        const float dmu = cut_f32(fma(-t, h[1], G)) / tf;
        if (fabsf(dmu) < 1e-9f) {
          g_shift(t, widen_f64(dmu), g0, h, g);
          if (kZ) z = z_of_t<EDF>(g[0]);
          return 0;
        }
      }
    }
  }
  return solve_z_from_n_theta_general<EDF>(n, theta, z, g);
}

// ------------------------------------------------------------ Landau frame
// T^a_b U^b = eps U^a (Eq. 21) written for U = gamma (1, u):
//   eps = T00 - m.u,   m_i - Pi_ij u_j = eps u_i,   m = (T01, T02), Pi = T^{ij},
// solved by Newton's method in u from the ideal conformal-fluid estimate
// (eps + P = x with 2 x^2 - 3 T00 x + |m|^2 = 0, u = m / x). The fixed point is
// the eigenvector the paper's power method converges to.
struct Frame {
  double eps, ux, uy, gamma;
  int st;
};

// Any state: FP64 Newton throughout.
static __device__ __noinline__ Frame landau_general(double E, double mx, double my, double pxx, double pxy, double pyy) {
  Frame F;
  F.eps = F.ux = F.uy = F.gamma = 0.0;
  F.st = ST_NONPHYSICAL;
  const double disc = 9.0 * E * E - 8.0 * (mx * mx + my * my);
  if (!(E > 0.0) || !(disc >= 0.0)) return F;
  const double x = 0.25 * (3.0 * E + sqrt(disc));
  double ux = mx / x, uy = my / x;
  int st = ST_LANDAU;
  for (int it = 0; it < 30; ++it) {
    const double a = E - (mx * ux + my * uy);
    const double fx = mx - (pxx * ux + pxy * uy) - a * ux;
    const double fy = my - (pxy * ux + pyy * uy) - a * uy;
    const double j00 = ux * mx - pxx - a, j01 = ux * my - pxy;
    const double j10 = uy * mx - pxy, j11 = uy * my - pyy - a;
    const double rdet = 1.0 / (j00 * j11 - j01 * j10);
    const double dx = (j01 * fy - j11 * fx) * rdet;
    const double dy = (j10 * fx - j00 * fy) * rdet;
    ux += dx;
    uy += dy;
    if (fmax(fabs(dx), fabs(dy)) < 1e-13) { st = 0; break; }
  }
  const double u2 = ux * ux + uy * uy;
  if (!(u2 < 1.0)) return F;
  F.ux = ux;
  F.uy = uy;
  F.eps = E - (mx * ux + my * uy);
  F.gamma = 1.0 / sqrt(1.0 - u2);
  if (F.eps > 0.0) F.st = st;
  return F;
}

// The same root with the iterations in FP32: Newton in FP32 (about 1e-7), then FP64
// residuals corrected through the FP32 Jacobian, whose 1e-6 only scales a correction,
// so two of them reach the FP64 floor (about 30 FP64 instructions against 270 for five
// FP64 steps). States near the light cone or out of the
// FP32 range, and any whose corrections do not shrink, take landau_general.
__device__ __forceinline__ int landau(const double T[6], Frame& F) {
  const float E = cut_f32(T[0]), mx = cut_f32(T[1]), my = cut_f32(T[2]), pxx = cut_f32(T[3]), pxy = cut_f32(T[4]),
              pyy = cut_f32(T[5]);
  const float disc = fmaf(9.0f * E, E, -8.0f * fmaf(mx, mx, my * my));
  if (E > 1e-15f && E < 1e15f && disc > 0.1f * E * E) {
    const float rx = 4.0f / fmaf(3.0f, E, sqrtf(disc));
    float fu = mx * rx, fv = my * rx, j00, j01, j10, j11, rdet;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const float a = fmaf(-mx, fu, fmaf(-my, fv, E));
      j00 = fmaf(fu, mx, -pxx) - a;
      j01 = fmaf(fu, my, -pxy);
      j10 = fmaf(fv, mx, -pxy);
      j11 = fmaf(fv, my, -pyy) - a;
      rdet = 1.0f / fmaf(j00, j11, -j01 * j10);
      if (it == 3) break;  // the Jacobian at the FP32 root
      const float fx = fmaf(-a, fu, fmaf(-pxx, fu, fmaf(-pxy, fv, mx)));
      const float fy = fmaf(-a, fv, fmaf(-pxy, fu, fmaf(-pyy, fv, my)));
      fu = fmaf(fmaf(j01, fy, -j11 * fx), rdet, fu);
      fv = fmaf(fmaf(j10, fx, -j00 * fy), rdet, fv);
    }
    if (fmaf(fu, fu, fv * fv) < 0.95f) {
      double ux = widen_f64(fu), uy = widen_f64(fv);
      float d = 0.0f;
      for (int it = 0; it < 6; ++it) {
        const double a = fma(-T[1], ux, fma(-T[2], uy, T[0]));
        const float fx = cut_f32(fma(-a, ux, fma(-T[3], ux, fma(-T[4], uy, T[1]))));
        const float fy = cut_f32(fma(-a, uy, fma(-T[4], ux, fma(-T[5], uy, T[2]))));
        const float dx = fmaf(j01, fy, -j11 * fx) * rdet, dy = fmaf(j10, fx, -j00 * fy) * rdet;
        ux += widen_f64(dx);
        uy += widen_f64(dy);
        d = fmaxf(fabsf(dx), fabsf(dy));
        if (d < 2e-11f) break;  // the next one would be below 1e-16
      }
      if (d < 2e-11f) {
        F.ux = ux;
        F.uy = uy;
        F.eps = fma(-T[1], ux, fma(-T[2], uy, T[0]));
        F.gamma = rsqrt64(fma(-ux, ux, fma(-uy, uy, 1.0)));
        if (!(F.eps > 0.0)) return ST_NONPHYSICAL;
        return 0;
      }
    }
  }
  F = landau_general(T[0], T[1], T[2], T[3], T[4], T[5]);
  return F.st;
}

// Macroscopic state of a cell: n = U_mu N^mu, theta, z (Eqs. 23-25).
struct CellState {
  double n, theta, ux, uy, z, eps, gamma;
  double g[6];
};

// The frame and n of a cell.
__device__ __forceinline__ int cell_frame(const double N[3], const double T[6], CellState& S) {
  Frame F;
  const int st = landau(T, F);
  if (st & ST_NONPHYSICAL) return st;
  S.ux = F.ux;
  S.uy = F.uy;
  S.gamma = F.gamma;
  S.eps = F.eps;
  S.n = F.gamma * fma(-F.ux, N[1], fma(-F.uy, N[2], N[0]));
  if (!(S.n > 0.0) || !isfinite(S.n) || !isfinite(S.eps)) return st | ST_NONPHYSICAL;
  return st;
}

// theta and the g_nu from n and eps. kZ: z is wanted (the read-out; a step only needs
// the g_nu).
template <int EDF, bool kZ>
__device__ __forceinline__ int cell_theta(CellState& S) {
  if (EDF == EDF_MJ) {
    S.theta = 0.5 * (S.eps * rcp64(S.n));
    if (kZ) {
      S.z = S.n / (2.0 * PI * S.theta * S.theta);
#pragma unroll
      for (int i = 0; i < 6; ++i) S.g[i] = S.z;
    }
    return 0;
  }
  const double rn = rcp64(S.n), en = S.eps * rn;
  const double target = (0.5 * PI) * (en * en * rn);
  const int zs = solve_z_from_R<EDF, kZ>(target, S.z, S.g);
  if (zs & ST_CLAMPED) S.theta = sqrt(S.n / (2.0 * PI * S.g[1]));
  else S.theta = 0.5 * (S.g[1] * rcp64(S.g[2])) * en;
  return zs;
}

template <int EDF, bool kZ>
__device__ __forceinline__ int cell_state(const double N[3], const double T[6], CellState& S) {
  int st = cell_frame(N, T, S);
  if (!(st & ST_NONPHYSICAL)) st |= cell_theta<EDF, kZ>(S);
  return st;
}

// --------------------------------------------- equilibrium moments (harmonic)
// Z_nk = int dp dphi f^eq p^n e^{i k phi} = Y_nk (u_x + i u_y)^k,
// Y_nk = 2 pi n! g_{n+1}(z) theta^{n+1} gamma^n P_nk(u^2),  k <= n <= 5: the real
// factors y, indexed n(n+1)/2 + k. The degree-1 and degree-2 prefactors are the
// cell's own n gamma and eps gamma^2 (2 pi g_2 theta^2 = n, 4 pi g_3 theta^3 = eps,
// Eq. 25), so that the collision conserves N^0 and T^{mu 0} without a rounding bias
// from the z, theta round trip; eps is the equilibrium's own energy. For MJ every
// g_nu is z, and the other prefactors follow from n, eps and theta alone.
// oi selects the expansion order's defect table (order - 2).
template <int EDF>
__device__ __forceinline__ void eq_moments(const double g[6], double theta, double u2, double gamma, double n,
                                           double eps, double y[21], int oi = kOrder5) {
  double A[6];
  const double tg = theta * gamma;
  A[1] = n * gamma;
  A[2] = eps * (gamma * gamma);
  if (EDF == EDF_MJ) {
    A[0] = n * rcp64(theta);
    A[3] = 3.0 * (tg * A[2]);
    A[4] = 4.0 * (tg * A[3]);
    A[5] = 5.0 * (tg * A[4]);
  } else {
    double q = (12.0 * PI) * (theta * tg) * (tg * tg);
    A[0] = (2.0 * PI) * (theta * g[0]);
    A[3] = q * g[3];
    q *= 4.0 * tg;
    A[4] = q * g[4];
    q *= 5.0 * tg;
    A[5] = q * g[5];
  }
#pragma unroll
  for (int n_ = 0; n_ < 6; ++n_)
#pragma unroll
    for (int k = 0; k <= n_; ++k) {
      const int i = n_ * (n_ + 1) / 2 + k;
      const double p0 = pnk(3 * i), p1 = pnk(3 * i + 1), p2 = pnk(3 * i + 2);
      if (p2 != 0.0) y[i] = A[n_] * fma(u2, fma(u2, p2, p1), p0);
      else if (p1 != 0.0) y[i] = A[n_] * fma(u2, p1, p0);
      else y[i] = p0 == 1.0 ? A[n_] : A[n_] * p0;
    }
  // The rounded projection table misses the identities that make the discrete
  // N^0, T^00 and T^0x, T^0y of f^eq equal Z_10, Z_20, Z_21 by the tiny constant
  // defects e1, e2, e3; correcting those three moments removes the resulting
  // bias (a constant error times Z would drift the conserved totals every step).
  // The corrections are below 2^-50 of the moments, so FP32 gives them to 2^-70.
  float Af[6], big = 0.0f;
  const float u2f = cut_f32(u2);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    Af[k] = cut_f32(A[k]);
    big = fmaxf(big, fabsf(Af[k]));
  }
  if (big < 1e30f && big > 1e-15f) {
    float d10 = 0.0f, d20 = 0.0f, d21 = 0.0f;
#pragma unroll
    for (int n_ = 0; n_ < 6; ++n_) {
#pragma unroll
      for (int k = 0; k <= (n_ ? 1 : 0); ++k) {
        const int i = 3 * (n_ * (n_ + 1) / 2 + k);
        const float yf = Af[n_] * fmaf(u2f, fmaf(u2f, (float)pnk(i + 2), (float)pnk(i + 1)), (float)pnk(i));
        if (k == 0) {
          d10 = fmaf(c_tf.e[oi][EDF][n_], yf, d10);
          d20 = fmaf(c_tf.e[oi][EDF][6 + n_], yf, d20);
        } else {
          d21 = fmaf(c_tf.e[oi][EDF][12 + n_], yf, d21);
        }
      }
    }
    y[1] -= widen_f64(d10);
    y[3] -= widen_f64(d20);
    y[4] -= widen_f64(d21);
  } else {  // moments outside the FP32 range
    double d10 = 0.0, d20 = 0.0, d21 = 0.0;
    for (int k = 0; k < 6; ++k) {
      d10 = fma(c_E[oi][EDF][k], y[k * (k + 1) / 2], d10);
      d20 = fma(c_E[oi][EDF][6 + k], y[k * (k + 1) / 2], d20);
      if (k) d21 = fma(c_E[oi][EDF][12 + k], y[k * (k + 1) / 2 + 1], d21);
    }
    y[1] -= d10;
    y[3] -= d20;
    y[4] -= d21;
  }
}

// C_k(d) = Re[(u_x + i u_y)^k e^{-i k phi_d}] of the directions d = 0..5 (d + 6
// flips the sign of odd k): C_2 flips and C_4 repeats after three directions, C_3
// is +-Re or +-Im (u_x + i u_y)^3. Computed once per cell, they replace the powers
// in every shell's synthesis (56 FP64 instructions per shell instead of 81, and
// C_1 is v_d . u, which the relaxation rate needs too).
struct DirPow {
  double c1[6], c5[6], c2[3], c4[3], w3r, w3i;
};

__device__ __forceinline__ DirPow dir_powers(double ux, double uy) {
  DirPow C;
  const double h = SQRT3_2;
  const double w2r = fma(ux, ux, -(uy * uy)), w2i = 2.0 * (ux * uy);
  C.w3r = fma(w2r, ux, -(w2i * uy));
  C.w3i = fma(w2r, uy, w2i * ux);
  const double w4r = fma(w2r, w2r, -(w2i * w2i)), w4i = 2.0 * (w2r * w2i);
  const double w5r = fma(w4r, ux, -(w4i * uy)), w5i = fma(w4r, uy, w4i * ux);
  // k = 1: angles 0, 30, .. 150; k = 5: 0, 150, 300, 90, 240, 30
  const double hx = h * ux, hy = h * uy, gx = h * w5r, gy = h * w5i;
  C.c1[0] = ux;
  C.c1[1] = fma(0.5, uy, hx);
  C.c1[2] = fma(0.5, ux, hy);
  C.c1[3] = uy;
  C.c1[4] = fma(-0.5, ux, hy);
  C.c1[5] = fma(0.5, uy, -hx);
  C.c5[0] = w5r;
  C.c5[1] = fma(0.5, w5i, -gx);
  C.c5[2] = fma(0.5, w5r, -gy);
  C.c5[3] = w5i;
  C.c5[4] = fma(-0.5, w5r, -gy);
  C.c5[5] = fma(0.5, w5i, gx);
  // k = 2: angles 0, 60, 120; k = 4: 0, 120, 240
  const double qy = h * w2i, ry = h * w4i;
  C.c2[0] = w2r;
  C.c2[1] = fma(0.5, w2r, qy);
  C.c2[2] = fma(-0.5, w2r, qy);
  C.c4[0] = w4r;
  C.c4[1] = fma(-0.5, w4r, ry);
  C.c4[2] = fma(-0.5, w4r, -ry);
  return C;
}

// Discrete equilibrium of one shell s at the 12 directions (order index oi =
// N - 2; the fifth order by default):
//   f^eq_{ds} = sum_k R_k C_k(d),  R_k = sum_{n>=k} Q^(k)_{s n} Y_nk,
// even k the same (E) and odd k of opposite sign (O) at d + 6.
template <int EDF>
__device__ __forceinline__ void shell_project(int s, const double y[21], double R[6], int oi = kOrder5) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double a = c_Q[oi][EDF][qoff(k) + s * (6 - k)] * y[k * (k + 1) / 2 + k];
#pragma unroll
    for (int n = k + 1; n < 6; ++n) a = fma(c_Q[oi][EDF][qoff(k) + s * (6 - k) + (n - k)], y[n * (n + 1) / 2 + k], a);
    R[k] = a;
  }
}

// E and O of direction d < 6; p3 = R_3 Re w^3, q3 = R_3 Im w^3 (C_3(d): Re, Im, -Re,
// -Im, Re, Im of w^3).
__device__ __forceinline__ void synth_dir(int d, const double R[6], double p3, double q3, const DirPow& C, double& E,
                                          double& O) {
  const double o3 = d % 2 ? (d == 3 ? -q3 : q3) : (d == 2 ? -p3 : p3);
  E = fma(d < 3 ? R[2] : -R[2], C.c2[d % 3], fma(R[4], C.c4[d % 3], R[0]));
  O = fma(R[1], C.c1[d], fma(R[5], C.c5[d], o3));
}

template <int EDF>
__device__ __forceinline__ void feq_shell(int s, const double y[21], const DirPow& C, double fe[12],
                                          int oi = kOrder5) {
  double R[6];
  shell_project<EDF>(s, y, R, oi);
  const double p3 = R[3] * C.w3r, q3 = R[3] * C.w3i;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    double E, O;
    synth_dir(d, R, p3, q3, C, E, O);
    fe[d] = E + O;
    fe[d + 6] = E - O;
  }
}

// ------------------------------------------------------------------ moments
// Harmonic sums of a 12-vector v over the directions: sum v, sum cos v,
// sum sin v, sum cos2 v, sum sin2 v (pairs d, d+6 folded first).
struct Harm {
  double h0, c1, s1, c2, s2;
};

__device__ __forceinline__ Harm harmonics_eo(const double e[6], const double o[6], bool need2) {
  const double h = SQRT3_2;
  Harm H;
  H.h0 = ((e[0] + e[1]) + (e[2] + e[3])) + (e[4] + e[5]);
  H.c1 = fma(h, o[1] - o[5], fma(0.5, o[2] - o[4], o[0]));
  H.s1 = fma(h, o[2] + o[4], fma(0.5, o[1] + o[5], o[3]));
  if (need2) {
    H.c2 = fma(0.5, (e[1] - e[2]) + (e[5] - e[4]), e[0] - e[3]);
    H.s2 = h * ((e[1] + e[2]) - (e[4] + e[5]));
  } else {
    H.c2 = H.s2 = 0.0;
  }
  return H;
}

__device__ __forceinline__ Harm harmonics(const double v[12], bool need2) {
  double e[6], o[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    e[d] = v[d] + v[d + 6];
    o[d] = v[d] - v[d + 6];
  }
  return harmonics_eo(e, o, need2);
}

// N^mu and T^{mu nu} from the harmonic sums of A_d and B_d.
__device__ __forceinline__ void moments_of(const Harm& ha, const Harm& hb, double N[3], double T[6]) {
  N[0] = ha.h0; N[1] = ha.c1; N[2] = ha.s1;
  T[0] = hb.h0; T[1] = hb.c1; T[2] = hb.s1;
  T[3] = 0.5 * (hb.h0 + hb.c2);
  T[4] = 0.5 * hb.s2;
  T[5] = 0.5 * (hb.h0 - hb.c2);
}

}  // namespace rlbm
