// Mixed-precision step: FP32 / BF16 / FP16 storage, FP32 streaming, equilibrium
// and relaxation carried out on deviations f - fref from each domain's rest
// reference equilibrium, and double-float (an unevaluated pair of FP32 numbers,
// about 48 bits) for the quantities that set conservation: the totals N^mu,
// T^{mu nu}, the Landau-frame residual (Eq. 21), gamma, n, eps and the degree-1
// and degree-2 equilibrium moments.
//
// GB300 executes FP64 at 1/64 of the FP32 rate, so the kernel issues no FP64
// instruction: the 72-term moment sums run in FP32 on the small deviations
// (their rounding error is relative to the deviation, not to f), the Landau
// solve is FP32 Newton followed by one correction with a double-float residual,
// and the equilibrium moments that the collision must reproduce exactly for N^0
// and T^{mu 0} (Z_1k = n gamma (u_x + i u_y)^k P_1k, Z_2k = eps gamma^2
// (u_x + i u_y)^k P_2k) are formed from the double-float n and eps.
//
// This header holds the kernels and their host helpers; each storage format is
// instantiated in a translation unit of its own (rlbm_mixed_<storage>.cu) so
// that the units compile in parallel, and rlbm_mixed.cu dispatches to them.
// Every unit that includes it has its own copy of the constant tables.
#pragma once
#include <cuda_runtime.h>

#include "rlbm_dfloat.cuh"
#include "rlbm_kernels.cuh"
#include "rlbm_tma.cuh"

namespace rlbm {

// ------------------------------------------------------------- FP32 tables
// terms of the power series of Li_nu(x), |x| <= 1/4 (the first one left out is below
// 2^-24 of g_1), of the expansions in ln z, of the series in t = g_1 and of the
// reversions t(w), t(G) (see solve_z_from_R)
constexpr int kSerF = 12, kExpBEf = 16, kExpFDf = 26, kLogSerF = 9, kRevF = RLBM_NREV;

// The FP64 tables rounded once to FP32 and laid out as the kernels read them, at
// compile time: the constant bank holds them when the library is loaded, and creating
// a handle uploads nothing.
struct MixedTables {
  float2 p[3][6];        // (p_s, p_s^2)
  // projection by shell pair: Qp[EDF][j][i] = Q^(k)_{s n} of s = 2j and 2j + 1, i = n(n+1)/2 + k
  float2 Qp[3][3][21];
  float E[3][18];        // exact defects of the FP32 tables in the conserved moments (see eq_moments)
  float2 invpow[3][kSerF];  // k^-nu of nu = 2i + 1, 2i + 2
  float be_exp[6 * kExpBEf], fd_exp[6 * kExpFDf];
  float be_logcoef[6], be_harm[6], g_zc[6];
  float logser[5 * kLogSerF], rev[kRevF], revg[kRevF];
};

constexpr MixedTables make_mixed_tables() {
  constexpr float pf[3][6] = {RLBM_PF_MJ_INIT, RLBM_PF_FD_INIT, RLBM_PF_BE_INIT};
  constexpr double p2[3][6] = {RLBM_P2_MJ_INIT, RLBM_P2_FD_INIT, RLBM_P2_BE_INIT};
  constexpr float Q[3][126] = {RLBM_QF_MJ_INIT, RLBM_QF_FD_INIT, RLBM_QF_BE_INIT};  // order k, s, n
  constexpr float E[3][18] = {RLBM_EF_MJ_INIT, RLBM_EF_FD_INIT, RLBM_EF_BE_INIT};
  constexpr double inv[6 * RLBM_NSERIES] = RLBM_INVPOW_INIT;
  constexpr double be[6 * RLBM_NEXP] = RLBM_BE_EXP_INIT;
  constexpr double fd[6 * RLBM_NEXP] = RLBM_FD_EXP_INIT;
  constexpr double lc[6] = RLBM_BE_LOGCOEF_INIT, hm[6] = RLBM_BE_HARM_INIT, gz[6] = RLBM_G_ZC_INIT;
  constexpr double ls[5 * RLBM_NLOGSER] = RLBM_LOGSER_INIT;
  constexpr double rv[RLBM_NREV] = RLBM_REV_INIT, rg[RLBM_NREV] = RLBM_REVG_INIT;
  MixedTables t{};
  for (int e = 0; e < 3; ++e) {
    for (int s = 0; s < 6; ++s) t.p[e][s] = float2{pf[e][s], (float)p2[e][s]};
    for (int i = 0; i < 18; ++i) t.E[e][i] = E[e][i];
    for (int j = 0; j < 3; ++j)
      for (int n = 0; n < 6; ++n)
        for (int k = 0; k <= n; ++k) {
          const int o = qoff(k) + (n - k);
          t.Qp[e][j][n * (n + 1) / 2 + k] = float2{Q[e][o + 2 * j * (6 - k)], Q[e][o + (2 * j + 1) * (6 - k)]};
        }
  }
  for (int nu = 0; nu < 6; ++nu) {
    for (int k = 0; k < kSerF; ++k) {
      const float v = (float)inv[nu * RLBM_NSERIES + k];
      if (nu % 2) t.invpow[nu / 2][k].y = v;
      else t.invpow[nu / 2][k].x = v;
    }
    for (int k = 0; k < kExpBEf; ++k) t.be_exp[nu * kExpBEf + k] = (float)be[nu * RLBM_NEXP + k];
    for (int k = 0; k < kExpFDf; ++k) t.fd_exp[nu * kExpFDf + k] = (float)fd[nu * RLBM_NEXP + k];
    t.be_logcoef[nu] = (float)lc[nu];
    t.be_harm[nu] = (float)hm[nu];
    t.g_zc[nu] = (float)gz[nu];
  }
  for (int nu = 0; nu < 5; ++nu)
    for (int k = 0; k < kLogSerF; ++k) t.logser[nu * kLogSerF + k] = (float)ls[nu * RLBM_NLOGSER + k];
  for (int k = 0; k < kRevF; ++k) {
    t.rev[k] = (float)rv[k];
    t.revg[k] = (float)rg[k];
  }
  return t;
}
static __constant__ MixedTables c_mt = make_mixed_tables();

constexpr float kPIf = 3.14159265358979f;
// sqrt(3)/2 = kH + kHl: FP32 value and its residual. Products with sqrt(3)/2
// take both parts (two FMAs): with kH alone every moment and synthesis that
// pairs directions at +-30 degrees would shrink by the same 1.8e-8 each step,
// a steady sink of momentum (a Taylor-Green flow decayed 1e-5 too fast in 500
// steps).
constexpr float kH = 0.866025403784438647f;
constexpr float kHl = (float)(0.866025403784438647 - (double)kH);
__device__ __forceinline__ float mul_h(float x) { return fmaf(kH, x, kHl * x); }
constexpr float kRZCf = (float)RLBM_R_ZC;
constexpr float kZCf = 0.9999999f;

// --------------------------------------------------- FP32 EDF integrals g_nu
// sum_{k>=1} x^k k^{-nu}, nu = 1..6, |x| <= 1/4, two nu as a pair. Fully unrolled, so
// that the coefficients are immediate constant operands. Rolled, each term loaded its
// six coefficients first; unrolling made the FD and BE steps 14 % and 5 % faster.
__device__ __forceinline__ void li_series6f(float x, float g[6]) {
  float xk = x;
  f2 a[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) a[i] = vmul(f2_dup(xk), f2_make(c_mt.invpow[i][0].x, c_mt.invpow[i][0].y));
#pragma unroll
  for (int k = 2; k <= kSerF; ++k) {
    xk *= x;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      a[i] = vfma(f2_dup(xk), f2_make(c_mt.invpow[i][k - 1].x, c_mt.invpow[i][k - 1].y), a[i]);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) f2_split(a[i], g[2 * i], g[2 * i + 1]);
}

template <int EDF>
__device__ void g_allf(float z, float g[6]) {
  if (EDF == EDF_MJ) {
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = z;
    return;
  }
  if (EDF == EDF_BE) {
    if (z <= 0.25f) { li_series6f(z, g); return; }
    const float mu = logf(z);
    float mk = 1.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = 0.0f;
#pragma unroll 4
    for (int k = 0; k < kExpBEf; ++k) {
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = fmaf(mk, c_mt.be_exp[i * kExpBEf + k], g[i]);
      mk *= mu;
    }
    const float lnm = logf(-mu);
    float mp = 1.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      g[i] = fmaf(mp, fmaf(-c_mt.be_logcoef[i], lnm, c_mt.be_harm[i]), g[i]);
      mp *= mu;
    }
    return;
  }
  if (z <= 0.25f) {
    li_series6f(-z, g);
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = -g[i];
    return;
  }
  if (z <= 4.0f) {
    const float mu = logf(z);
    float mk = 1.0f;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = 0.0f;
#pragma unroll 2
    for (int k = 0; k < kExpFDf; ++k) {
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = fmaf(mk, c_mt.fd_exp[i * kExpFDf + k], g[i]);
      mk *= mu;
    }
    return;
  }
  li_series6f(-1.0f / z, g);
  const float L = logf(z);
  const float eta2 = 0.822467033f, eta4 = 0.947032829f, eta6 = 0.985551091f;
  const float L2 = L * L, L3 = L2 * L, L4 = L3 * L, L5 = L4 * L, L6 = L5 * L;
  // the inversion formula's polynomial in L, products and sums written out
  g[0] = -g[0] + L;
  g[1] = g[1] + fmaf(L2, 0.5f, 2.0f * eta2);
  g[2] = -g[2] + fmaf(L3, 1.0f / 6.0f, (2.0f * eta2) * L);
  g[3] = g[3] + fmaf(L4, 1.0f / 24.0f, fmaf(eta2, L2, 2.0f * eta4));
  g[4] = -g[4] + fmaf(L5, 1.0f / 120.0f, fmaf(eta2 / 3.0f, L3, (2.0f * eta4) * L));
  g[5] = g[5] + fmaf(L6, 1.0f / 720.0f, fmaf(eta2 / 12.0f, L4, fmaf(eta4, L2, 2.0f * eta6)));
}

// g_1, g_2, g_3 alone (g[0..2] of g_allf), what the Newton iterations below
// need: in the series range three series instead of six.
template <int EDF>
__device__ __forceinline__ void g123f(float z, float g[3]) {
  if (EDF != EDF_MJ && z <= 0.25f) {
    const float x = EDF == EDF_BE ? z : -z;
    float xk = x, s1, s2, s3 = xk * c_mt.invpow[1][0].x;
    f2 a = vmul(f2_dup(xk), f2_make(c_mt.invpow[0][0].x, c_mt.invpow[0][0].y));
#pragma unroll
    for (int k = 2; k <= kSerF; ++k) {
      xk *= x;
      a = vfma(f2_dup(xk), f2_make(c_mt.invpow[0][k - 1].x, c_mt.invpow[0][k - 1].y), a);
      s3 = fmaf(xk, c_mt.invpow[1][k - 1].x, s3);
    }
    f2_split(a, s1, s2);
    const float sg = EDF == EDF_BE ? 1.0f : -1.0f;
    g[0] = sg * s1;
    g[1] = sg * s2;
    g[2] = sg * s3;
    return;
  }
  float g6[6];
  g_allf<EDF>(z, g6);
  g[0] = g6[0];
  g[1] = g6[1];
  g[2] = g6[2];
}

// A Newton step d in mu leaves an error of about C d^2, with C = |F''/(2F')| of
// the equation solved. Computed with arbitrary-precision polylogs, C is at most
// 0.23 for FD (z from 0.17 to 30) and about 0.12/(1 - z) for BE (0.24 at
// z = 0.5, 13 at z = 0.99), for both solves below. So a Newton step with
// d^2 C_bound < 1e-9 (C_bound = 0.25, or 0.25/(1 - z) for BE) is accepted
// without evaluating the equation again: the result is within 1e-9 of the root.
template <int EDF>
__device__ __forceinline__ bool newton_done(float d, float z) {
  const float cb = EDF == EDF_BE ? 0.25f / (1.0f - z) : 0.25f;
  return d * d * cb < 1e-9f;
}

// The six g_nu of t = g_1 <= 0.5 (z = 0.65 FD, 0.39 BE): nine terms put the first one
// left out below 1e-9 of the sum; no logarithm, no exponential (see h_all_t).
template <int EDF>
__device__ __forceinline__ void g_all_tf(float t, float g[6]) {
  const float u = EDF == EDF_BE ? t : -t, u2 = u * u;
  float a = c_mt.logser[8], b[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j] = c_mt.logser[(j + 1) * kLogSerF + 8];
  a = fmaf(fmaf(fmaf(a, u2, c_mt.logser[6]), u2, c_mt.logser[4]), u2, c_mt.logser[2]);  // odd ones vanish
#pragma unroll
  for (int n = 7; n >= 0; --n)
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = fmaf(b[j], u, c_mt.logser[(j + 1) * kLogSerF + n]);
  g[0] = t;
  g[1] = t * fmaf(a, u2, fmaf(u, -0.25f, 1.0f));
#pragma unroll
  for (int j = 0; j < 4; ++j) g[2 + j] = t * b[j];
}
template <int EDF>
__device__ __forceinline__ float z_of_tf(float t) { return EDF == EDF_BE ? -expm1f(-t) : expm1f(t); }
// t = x sum_n a_n (s x)^n
template <int EDF>
__device__ __forceinline__ float revert_f(const float* c, float x) {
  const float sx = EDF == EDF_BE ? x : -x;
  float p = c[kRevF - 1];
#pragma unroll
  for (int n = kRevF - 2; n >= 0; --n) p = fmaf(p, sx, c[n]);
  return x * p;
}

// Fugacity from g_3^2/g_2^3 = target (Eq. 25), FP32 safeguarded Newton in mu = ln z.
// Start: the series g_nu = z + s z^2/2^nu + z^3/3^nu + s z^4/4^nu ... (s = -1 FD,
// +1 BE) make w = 1/target = g_2^3/g_3^2 a power series in z; inverting it gives
// mu = ln w - s w/2 + (119/1728) w^2 - s (85/6912) w^3 + O(w^4), off by 1.4e-6 in
// mu at z = 0.17, so one Newton step reaches the FP32 floor (newton_done accepts
// it). The iterations evaluate g_1..g_3 alone; all six g_nu are evaluated once,
// at the converged mu (the last step applied).
template <int EDF>
__device__ __forceinline__ int solve_z_R_newton_f(float target, float& z, float g[6]) {
  if (EDF == EDF_BE && target < kRZCf) {
    z = kZCf;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = c_mt.g_zc[i];
    return ST_CLAMPED;
  }
  float lo = -40.0f, hi = (EDF == EDF_BE) ? -1.0e-7f : 40.0f;
  const float lt = logf(target);
  float mu = -lt;
  {
    const float w = 1.0f / target;
    if (w < 0.5f) {
      constexpr float kS = EDF == EDF_BE ? 1.0f : -1.0f;
      mu = fmaf(fmaf(fmaf(-kS * (85.0f / 6912.0f), w, 119.0f / 1728.0f), w, -0.5f * kS), w, mu);
    }
  }
  mu = fminf(fmaxf(mu, lo + 1e-3f), hi);
  int st = ST_ZSOLVE;
  float dprev = INFINITY;
  for (int it = 0; it < 40; ++it) {
    float gi[3];
    const float ze = expf(mu);
    g123f<EDF>(ze, gi);
    const float F = logf(gi[2] * gi[2] / (gi[1] * gi[1] * gi[1])) - lt;
    if (F == 0.0f) {
      st = 0;
      break;
    }
    const float dF = 2.0f * gi[1] / gi[2] - 3.0f * gi[0] / gi[1];
    if (F > 0.0f) lo = mu; else hi = mu;
    float mn = mu - F / dF;
    const bool newton = mn >= lo && mn <= hi;
    if (!newton) mn = 0.5f * (lo + hi);
    const float d = fabsf(mn - mu);
    mu = mn;
    if (d <= 4e-7f * fmaxf(1.0f, fabsf(mu)) || (newton && newton_done<EDF>(d, ze)) ||
        (d < 1e-4f && d >= dprev)) {
      st = 0;
      break;
    }
    dprev = d;
  }
  z = expf(mu);
  g_allf<EDF>(z, g);
  return st;
}

// Fugacity from (n, theta): n = 2 pi theta^2 g_2(z), FP32 safeguarded Newton in
// mu = ln z. Start: inverting G = g_2(z) = z -+ z^2/4 + z^3/9 -+ ... (G = n / (2 pi
// theta^2)) gives mu = ln G +- G/4 - (5/288) G^2 +- G^3/288 + O(G^4) (upper signs
// FD, lower BE) for small G. Convergence as in solve_z_R_f.
template <int EDF>
__device__ __forceinline__ int solve_z_nt_newton_f(float n, float theta, float& z, float g[6]) {
  const float G = n / (2.0f * kPIf * theta * theta);
  if (EDF == EDF_BE && G >= c_mt.g_zc[1]) {
    z = kZCf;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = c_mt.g_zc[i];
    return ST_CLAMPED;
  }
  float lo = -40.0f, hi = (EDF == EDF_BE) ? -1.0e-7f : 40.0f;
  const float lG = logf(G);
  float mu = lG;
  if (G < 0.5f) {
    constexpr float kS = EDF == EDF_BE ? -1.0f : 1.0f;
    mu = fmaf(fmaf(fmaf(kS / 288.0f, G, -5.0f / 288.0f), G, 0.25f * kS), G, mu);
  }
  mu = fminf(fmaxf(mu, lo + 1e-3f), hi);
  float dprev = INFINITY;
  int st = ST_ZSOLVE;
  for (int it = 0; it < 40; ++it) {
    float gi[3];
    const float ze = expf(mu);
    g123f<EDF>(ze, gi);
    const float F = logf(gi[1]) - lG;
    if (F == 0.0f) {
      st = 0;
      break;
    }
    const float dF = gi[0] / gi[1];
    if (F < 0.0f) lo = mu; else hi = mu;
    float mn = mu - F / dF;
    const bool newton = mn >= lo && mn <= hi;
    if (!newton) mn = 0.5f * (lo + hi);
    const float d = fabsf(mn - mu);
    mu = mn;
    if (d <= 4e-7f * fmaxf(1.0f, fabsf(mu)) || (newton && newton_done<EDF>(d, ze)) ||
        (d < 1e-4f && d >= dprev)) {
      st = 0;
      break;
    }
    dprev = d;
  }
  z = expf(mu);
  g_allf<EDF>(z, g);
  return st;
}

// Fugacity of a cell from n and eps, by the Newton solve on the target ratio; with
// kSeries (the 16-bit storages) from w = g_2^3/g_3^2 = (2/pi) n^3/eps^2. For w up to
// 0.48 (z about 0.61 FD, 0.38 BE) ten terms of the reversion t(w) = w + (47/1728) w^3 + ...
// give t to FP32 rounding (the first one left out is below 3e-9 of t) and g_all_tf
// the g_nu; other states take the Newton solve, out of line. kZ: z is wanted.
template <int EDF>
__device__ __noinline__ int solve_z_R_other_f(float target, float& z, float g[6]) {
  return solve_z_R_newton_f<EDF>(target, z, g);
}
template <int EDF>
__device__ __noinline__ int solve_z_nt_other_f(float n, float theta, float& z, float g[6]) {
  return solve_z_nt_newton_f<EDF>(n, theta, z, g);
}
template <int EDF, bool kSeries, bool kZ>
__device__ __forceinline__ int solve_z_R_f(float n, float eps, float& z, float g[6]) {
  const float target = 0.5f * kPIf * eps * eps / (n * n * n);
  if constexpr (kSeries) {
    const float w = (2.0f / kPIf) * (n * n * n) / (eps * eps);
    if (w > 1e-30f && w < 0.48f) {
      const float t = revert_f<EDF>(c_mt.rev, w);
      g_all_tf<EDF>(t, g);
      if (kZ) z = z_of_tf<EDF>(t);
      return 0;
    }
    return solve_z_R_other_f<EDF>(target, z, g);
  } else {
    return solve_z_R_newton_f<EDF>(target, z, g);
  }
}

// Fugacity from (n, theta): G = n / (2 pi theta^2) = g_2. The reversion t(G) converges
// more slowly (ratio about G/2): ten terms reach FP32 rounding up to G = 0.25.
template <int EDF, bool kSeries, bool kZ>
__device__ __forceinline__ int solve_z_nt_f(float n, float theta, float& z, float g[6]) {
  const float G = n / (2.0f * kPIf * theta * theta);
  if constexpr (EDF == EDF_MJ) {
    z = G;
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = G;
    return 0;
  } else if constexpr (kSeries) {
    if (G > 1e-30f && G < 0.25f) {
      const float t = revert_f<EDF>(c_mt.revg, G);
      g_all_tf<EDF>(t, g);
      if (kZ) z = z_of_tf<EDF>(t);
      return 0;
    }
    return solve_z_nt_other_f<EDF>(n, theta, z, g);
  } else {
    return solve_z_nt_newton_f<EDF>(n, theta, z, g);
  }
}

// ------------------------------------------------------------- Landau frame
// Moments of a cell: N0, m = (T^01, T^02) and c = (N^1, N^2) (the reference state has
// none), T^00 and the spatial stresses.
struct MomentsDf {
  df N0, T00, T11, T22;
  f2 nv, m;   // (N^1, N^2), (T^01, T^02)
  float T12;
};

// T^a_b U^b = eps U^a (Eq. 21) as m - Pi u = (T00 - m.u) u. FP32 Newton from the
// ideal-fluid estimate, then one Newton correction whose residual is evaluated
// in double-float (the FP32 Jacobian only scales the small correction), which
// brings u to ~1e-15. eps, gamma follow in double-float, |u|^2 and n on the way. The
// x and y components run as one pair.
struct FrameDf {
  df2 u;
  df eps, gamma, u2, n;
};

__device__ __forceinline__ int landau_df(const MomentsDf& M, FrameDf& F) {
  // every product that meets a sum is an explicit FMA (or the sum a rounded
  // intrinsic), so each kernel that inlines this gets the same roundings
  float mx, my;
  f2_split(M.m, mx, my);
  const float E = M.T00.hi, pxx = M.T11.hi, pxy = M.T12, pyy = M.T22.hi;
  const float disc = fmaf(9.0f * E, E, -8.0f * fmaf(mx, mx, __fmul_rn(my, my)));
  if (!(E > 0.0f) || !(disc >= 0.0f)) return ST_NONPHYSICAL;
  const float x = 0.25f * fmaf(3.0f, E, sqrtf(disc));
  float fu = mx / x, fv = my / x;
#pragma unroll
  for (int it = 0; it < 3; ++it) {
    const float a = fmaf(-mx, fu, fmaf(-my, fv, E));
    const float fx = fmaf(-a, fu, fmaf(-pxx, fu, fmaf(-pxy, fv, mx)));
    const float fy = fmaf(-a, fv, fmaf(-pxy, fu, fmaf(-pyy, fv, my)));
    const float j00 = __fsub_rn(fmaf(fu, mx, -pxx), a), j01 = fmaf(fu, my, -pxy), j10 = fmaf(fv, mx, -pxy),
                j11 = __fsub_rn(fmaf(fv, my, -pyy), a);
    const float rdet = 1.0f / fmaf(j00, j11, -__fmul_rn(j01, j10));
    fu = fmaf(fmaf(j01, fy, -__fmul_rn(j11, fx)), rdet, fu);
    fv = fmaf(fmaf(j10, fx, -__fmul_rn(j00, fy)), rdet, fv);
  }
  if (!(fmaf(fu, fu, __fmul_rn(fv, fv)) < 1.0f)) return ST_NONPHYSICAL;
  const f2 f = f2_make(fu, fv);
  {
    const df2 mf = two_prod(M.m, f);
    const df a = df_sub(M.T00, df_add(df_first(mf), df_second(mf)));
    const df2 pu = df_add(df_mul(df_make(f2_make(M.T11.hi, pxy), f2_make(M.T11.lo, 0.0f)), f2_dup(fu)),
                          df_mul(df_make(f2_make(pxy, M.T22.hi), f2_make(0.0f, M.T22.lo)), f2_dup(fv)));
    const df2 r = df_sub(df_add(df_neg(pu), M.m), df_mul(df_dup(a), f));
    const float af = a.hi;
    const float j00 = __fsub_rn(fmaf(fu, mx, -pxx), af), j01 = fmaf(fu, my, -pxy), j10 = fmaf(fv, mx, -pxy),
                j11 = __fsub_rn(fmaf(fv, my, -pyy), af);
    const float rdet = 1.0f / fmaf(j00, j11, -__fmul_rn(j01, j10));
    float gx, gy;
    f2_split(df_to_float(r), gx, gy);
    F.u = two_sum(f, f2_make(__fmul_rn(fmaf(j01, gy, -__fmul_rn(j11, gx)), rdet),
                             __fmul_rn(fmaf(j10, gx, -__fmul_rn(j00, gy)), rdet)));
  }
  const df2 mu = df_mul(F.u, M.m), uu = df_mul(F.u, F.u), nu = df_mul(F.u, M.nv);
  F.eps = df_sub(M.T00, df_add(df_first(mu), df_second(mu)));
  F.u2 = df_add(df_first(uu), df_second(uu));
  const df w = df_sub(df_make(1.0f, 0.0f), F.u2);
  if (!(w.hi > 0.0f) || !(F.eps.hi > 0.0f)) return ST_NONPHYSICAL;
  F.gamma = df_rsqrt(w);
  F.n = df_mul(F.gamma, df_sub(M.N0, df_add(df_first(nu), df_second(nu))));
  if (!(F.n.hi > 0.0f) || !isfinite(F.n.hi)) return ST_NONPHYSICAL;
  return 0;
}

// FP32 harmonic sums of the per-direction sums (A_d, B_d), the two kinds as a pair
// (directions d, d + 6 folded first), and the moment totals in double-float:
// reference moments + FP32 deviation sums.
__device__ __forceinline__ MomentsDf moments_df(const DomDev& D, const f2 v[12]) {
  const f2 half = f2_dup(0.5f), h = f2_dup(kH), hl = f2_dup(kHl);
  f2 e[6], o[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    e[d] = vadd(v[d], v[d + 6]);
    o[d] = vsub(v[d], v[d + 6]);
  }
  const f2 h0 = vadd(vadd(vadd(e[0], e[1]), vadd(e[2], e[3])), vadd(e[4], e[5]));
  const f2 c1x = vsub(o[1], o[5]), s1x = vadd(o[2], o[4]);
  const f2 c1 = vfma(h, c1x, vfma(hl, c1x, vfma(half, vsub(o[2], o[4]), o[0])));
  const f2 s1 = vfma(h, s1x, vfma(hl, s1x, vfma(half, vadd(o[1], o[5]), o[3])));
  float be[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) be[d] = f2_hi(e[d]);
  const float c2 = fmaf(0.5f, __fadd_rn(__fsub_rn(be[1], be[2]), __fsub_rn(be[5], be[4])), __fsub_rn(be[0], be[3]));
  const float s2 = mul_h(__fsub_rn(__fadd_rn(be[1], be[2]), __fadd_rn(be[4], be[5])));
  MomentsDf M;
  M.N0 = df_add(df_make(D.n0_hl[0], D.n0_hl[1]), f2_lo(h0));
  M.T00 = df_add(df_make(D.t00_hl[0], D.t00_hl[1]), f2_hi(h0));
  M.nv = f2_make(f2_lo(c1), f2_lo(s1));
  M.m = f2_make(f2_hi(c1), f2_hi(s1));
  M.T11 = df_scale(df_add(M.T00, c2), 0.5f);
  M.T12 = 0.5f * s2;
  M.T22 = df_scale(df_add(M.T00, -c2), 0.5f);
  return M;
}

// Relaxation rates gamma (1 - v_d . u) / tau (Eq. 3), the directions d and d + 6
// (v_d . u of opposite sign) as a pair, with the roundings written out (see landau_df).
__device__ __forceinline__ void relax_rates(float gam, float ux, float uy, float itau, float om[12]) {
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const float vu = fmaf((float)dcos(d), ux, __fmul_rn((float)dsin(d), uy));
    f2_split(vmul(vmul(f2_dup(gam), vsub(f2_dup(1.0f), f2_make(vu, -vu))), f2_dup(itau)), om[d], om[d + 6]);
  }
}

// Equilibrium-moment deviations dZ_nk = Z_nk - Z_ref, Re and Im, indexed n(n+1)/2 + k.
struct EqF {
  float zr[21], zi[21];
};

// FP32 deviation of the equilibrium from fref for the shells s = 2j, 2j + 1 (12
// directions, the two shells as a pair): R^{c|s}_k = sum_n Q^(k)_{s n} dZ_nk (+ rres_s in
// R^c_0), then the folded 12-point synthesis (same symmetries as the FP64 form). The
// harmonics carry the powers of u before the projection: the momentum of the
// equilibrium is a sum of Q Z_n1, whose rounding must vary from cell to cell with u
// (rounded as one constant factor times u it would be off by the same 3e-8 in every
// cell and step, a steady source of momentum).
template <int EDF>
__device__ __forceinline__ void dfeq_pair(int j, f2 rres, const EqF& q, f2 fe[12]) {
  f2 Rc[6], Rs[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
#pragma unroll
    for (int n = k; n < 6; ++n) {
      const int i = n * (n + 1) / 2 + k;
      const f2 t = f2_make(c_mt.Qp[EDF][j][i].x, c_mt.Qp[EDF][j][i].y);
      Rc[k] = n == k ? vmul(t, f2_dup(q.zr[i])) : vfma(t, f2_dup(q.zr[i]), Rc[k]);
      if (k) Rs[k] = n == k ? vmul(t, f2_dup(q.zi[i])) : vfma(t, f2_dup(q.zi[i]), Rs[k]);
    }
  }
  Rc[0] = vadd(Rc[0], rres);
  const f2 half = f2_dup(0.5f), mhalf = f2_dup(-0.5f), h = f2_dup(kH), hl = f2_dup(kHl);
  auto mulh = [&](f2 x) { return vfma(h, x, vmul(hl, x)); };
  const f2 t1 = vadd(Rc[0], Rc[4]), t2 = vfma(mhalf, Rc[4], Rc[0]);
  const f2 Ec0 = vadd(t1, Rc[2]), Ec3 = vsub(t1, Rc[2]), Ec1 = vfma(half, Rc[2], t2), Ec2 = vfma(mhalf, Rc[2], t2);
  const f2 Es1 = mulh(vadd(Rs[2], Rs[4])), Es2 = mulh(vsub(Rs[2], Rs[4]));
  const f2 E[6] = {Ec0, vadd(Ec1, Es1), vadd(Ec2, Es2), Ec3, vsub(Ec2, Es2), vsub(Ec1, Es1)};
  const f2 Oc0 = vadd(vadd(Rc[1], Rc[3]), Rc[5]), Oc1 = mulh(vsub(Rc[1], Rc[5])),
           Oc2 = vfma(half, vadd(Rc[1], Rc[5]), vneg(Rc[3]));
  const f2 Os1 = vfma(half, vadd(Rs[1], Rs[5]), Rs[3]), Os2 = mulh(vsub(Rs[1], Rs[5])),
           Os3 = vadd(vsub(Rs[1], Rs[3]), Rs[5]);
  const f2 O[6] = {Oc0, vadd(Oc1, Os1), vadd(Oc2, Os2), Os3, vsub(Os2, Oc2), vsub(Os1, Oc1)};
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    fe[d] = vadd(E[d], O[d]);
    fe[d + 6] = vsub(E[d], O[d]);
  }
}

// FP32 equilibrium-moment deviations dZ_nk = Z_nk - Z_ref (Appendix, harmonic
// form). When An1, An2 >= 0 they replace the degree-1 and degree-2 prefactors
// (n gamma and eps gamma^2 from the double-float state); the caller then sets
// the conserved isotropic entries dZ_10, dZ_20 itself.
template <int EDF>
__device__ __forceinline__ void dz_moments(const DomDev& D, const float g[6], float theta, float ux, float uy,
                                           float gam, float An1, float An2, EqF& q) {
  // products that meet sums are explicit FMAs (see landau_df)
  const float u2 = fmaf(ux, ux, __fmul_rn(uy, uy));
  float wr[6], wi[6];
  wr[1] = ux;
  wi[1] = uy;
#pragma unroll
  for (int k = 2; k < 6; ++k) {
    wr[k] = fmaf(wr[k - 1], ux, -__fmul_rn(wi[k - 1], uy));
    wi[k] = fmaf(wr[k - 1], uy, __fmul_rn(wi[k - 1], ux));
  }
  float A = 2.0f * kPIf * theta;
#pragma unroll
  for (int n = 0; n < 6; ++n) {
    if (n > 0) A = __fmul_rn(A, __fmul_rn(__fmul_rn((float)n, theta), gam));
    float An = __fmul_rn(A, g[n]);  // (a plain product would be contracted where P is 1)
    if (n == 1 && An1 >= 0.0f) An = An1;
    if (n == 2 && An2 >= 0.0f) An = An2;
#pragma unroll
    for (int k = 0; k <= n; ++k) {
      const int i = n * (n + 1) / 2 + k;
      const float p0 = (float)pnk(3 * i), p1 = (float)pnk(3 * i + 1), p2 = (float)pnk(3 * i + 2);
      const float P = p2 != 0.0f ? fmaf(u2, fmaf(u2, p2, p1), p0) : (p1 != 0.0f ? fmaf(u2, p1, p0) : p0);
      if (k == 0) {
        q.zr[i] = fmaf(An, P, -D.zref_f[n]);  // the isotropic moments as deviations from the reference
      } else {
        const float sc = __fmul_rn(An, P);
        q.zr[i] = __fmul_rn(sc, wr[k]);
        q.zi[i] = __fmul_rn(sc, wi[k]);
      }
    }
  }
}

// Remove the FP32 tables' defects in N^0, T^00, T^0x, T^0y (FP32 suffices: the
// corrections are ~1e-8 of the moments).
template <int EDF>
__device__ __forceinline__ void remove_defects(EqF& q) {
  float d10 = 0.0f, d20 = 0.0f, d21r = 0.0f, d21i = 0.0f;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    d10 = fmaf(c_mt.E[EDF][k], q.zr[k * (k + 1) / 2], d10);
    d20 = fmaf(c_mt.E[EDF][6 + k], q.zr[k * (k + 1) / 2], d20);
  }
#pragma unroll
  for (int k = 1; k < 6; ++k) {
    d21r = fmaf(c_mt.E[EDF][12 + k], q.zr[k * (k + 1) / 2 + 1], d21r);
    d21i = fmaf(c_mt.E[EDF][12 + k], q.zi[k * (k + 1) / 2 + 1], d21i);
  }
  q.zr[1] = __fsub_rn(q.zr[1], d10);
  q.zr[3] = __fsub_rn(q.zr[3], d20);
  q.zr[4] = __fsub_rn(q.zr[4], d21r);
  q.zi[4] = __fsub_rn(q.zi[4], d21i);
}

// Equilibrium deviations of a shell pair in work units (see the storage policies).
template <int EDF, class S>
__device__ __forceinline__ void dfeq_work(const DomDev& D, int j, const EqF& q, f2 fe[12]) {
  dfeq_pair<EDF>(j, f2_make(D.rres[2 * j], D.rres[2 * j + 1]), q, fe);
  if constexpr (S::kScaled) {
    const f2 b = f2_make(D.b_s[2 * j], D.b_s[2 * j + 1]);
#pragma unroll
    for (int d = 0; d < 12; ++d) fe[d] = vmul(b, fe[d]);
  }
}

// Halo writer of the mixed step: copies of the cell's post-collision values
// (work units, held in its shared-memory column col[pair * kThreads]) and, at
// fixed-T walls, the
// FP32 equilibrium deviation of the wall ghost. Reading the copies back from
// global memory instead would put a read-after-write round trip to L2 on every
// edge warp, which costs more than keeping the column up to date.
template <int EDF, class S>
__device__ __noinline__ void write_halo_mixed(const DomDev& D, int x, int y, typename S::T* __restrict__ fout,
                                              const f2* col, bool have_state, float n, float ux, float uy,
                                              float gam, unsigned& st, bool images) {
  using P = Pair<typename S::T>;
  int hx[8], hy[8], wall[8];
  const int cnt = halo_targets(D, x, y, hx, hy, wall, images);
  for (int i = 0; i < cnt; ++i) {
    typename S::T* h = fout + cell_rel(D, hx[i], hy[i]);
    if (wall[i] < 0 || !have_state) {
      for (int k = 0; k < kPairs; ++k)
        *reinterpret_cast<P*>(h + k * kSegW) = S::enc2(col[k * kThreads], D, 2 * (k % 3));
    } else {
      const float tw = D.t_wall_f[wall[i]];
      float z, g[6];
      st |= solve_z_nt_f<EDF, S::kScaled, false>(n, tw, z, g);
      EqF q;
      dz_moments<EDF>(D, g, tw, ux, uy, gam, -1.0f, -1.0f, q);
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        f2 fe[12];
        dfeq_work<EDF, S>(D, j, q, fe);
#pragma unroll
        for (int d = 0; d < 12; ++d) *reinterpret_cast<P*>(h + (3 * d + j) * kSegW) = S::enc2(fe[d], D, 2 * j);
      }
    }
  }
}

constexpr size_t kSmemF = 72 * kThreads * sizeof(float);  // the shared-memory column of a block

// Resident blocks of 128 threads per SM that the register budget must allow: 5 (96
// registers, 20 warps) for the FP32 storages without halo work, 4 (128 registers, 16
// warps) for the 16-bit ones and wherever the halo writer's arguments would spill.
// Measured, 5 against 4 blocks, MLUPS: 2048^2 FP32 deviations 11,096 / 10,919, 128-domain
// batch 10,734 / 10,514; the batch in FP16 12,322 / 12,600; FD Fourier batch with
// walls in BF16 8,558 / 10,427, in FP32 deviations 8,311 / 9,557.
template <class S, int kHalo>
constexpr int mixed_min_blocks() {
  return (kHalo == 0 && !S::kScaled ? 640 : 512) / kThreads;
}
// 1: at the start of a tile one thread asks L2 for the tile's own blocks in rows
// y0-1 .. y0+kTileH (one contiguous segment per row), so that the pull's later
// directions find them in L2
#ifndef RLBM_MIXED_L2_PREFETCH
#define RLBM_MIXED_L2_PREFETCH 1
#endif

// Relaxation (Eq. 3) of one cell's 72 pulled deviations in its column, a shell pair
// at a time (unrolled: the tables are immediate operands, 5 % faster than a loop),
// stored to fout; kKeep: the relaxed values also go back into the
// column (the halo writer reads them there).
template <int EDF, class S, bool kKeep>
__device__ __forceinline__ void relax_cell(const DomDev& D, const EqF& q, const float om[12], f2* col,
                                           typename S::T* __restrict__ out) {
  using P = Pair<typename S::T>;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    f2 fe[12];
    dfeq_work<EDF, S>(D, j, q, fe);
#pragma unroll
    for (int d = 0; d < 12; ++d) {
      const int k = 3 * d + j;
      const f2 v = col[k * kThreads];
      const f2 r = vfma(f2_dup(om[d]), vsub(fe[d], v), v);
      if constexpr (kKeep) col[k * kThreads] = r;
      *reinterpret_cast<P*>(out + k * kSegW) = S::enc2(r, D, 2 * j);
    }
  }
}

// Collision of one cell (Eqs. 20-25, 10-11 and 3) from its pulled values in work
// units, held in the thread's shared-memory column col[pair * kThreads],
// and the shell sums A_d = sum_s p_s dv_{6d+s}, B_d = sum_s p_s^2 dv_{6d+s} of
// each direction; stores f* to fout, writes the cell's halo images and returns
// its status bits. Called by the active lanes of a warp (the lanes of cells
// inside the domain). kImages: also write the periodic halo images (the
// TMA-staged step reads them; the L1 pull wraps instead). kHalo, the launch's
// halo work (StepArgs::halo): 0 none (every side periodic or exchanged), 1 wall
// equilibria only (every other side a fixed-T wall), 2 also copies (zero-gradient
// sides). Below 2, with kImages = false, no halo cell copies the cell's relaxed
// values, so they need not go back to the column.
template <int EDF, class S, bool kImages, int kHalo = 2>
__device__ __forceinline__ unsigned collide_mixed(const DomDev& D, int x, int y, long long c, const f2 AB[12],
                                                  f2* col, typename S::T* __restrict__ fout) {
  // a warp with no cell on an edge that has halo cells to write skips the halo
  // writer (uniform per warp)
  const bool edge = kImages ? (x == 0 || x == D.nx - 1 || y == 0 || y == D.ny - 1)
                            : kHalo > 0 && ((x == 0 && bc_writes_halo(D.bc[0])) ||
                                        (x == D.nx - 1 && bc_writes_halo(D.bc[1])) ||
                                        (y == 0 && bc_writes_halo(D.bc[2])) ||
                                        (y == D.ny - 1 && bc_writes_halo(D.bc[3])));
  const bool edge_warp = __any_sync(__activemask(), edge);
  const MomentsDf M = moments_df(D, AB);
  FrameDf F;
  unsigned st = landau_df(M, F);
  const bool ok = !(st & ST_NONPHYSICAL);
  float uxf = 0.0f, uyf = 0.0f, gf = 0.0f, nf = 0.0f;
  if (ok) {
    f2_split(df_to_float(F.u), uxf, uyf);
    gf = df_to_float(F.gamma);
    nf = df_to_float(F.n);
    const float ef = df_to_float(F.eps);
    float theta, z, g[6];
    if (EDF == EDF_MJ) {
      theta = ef / (2.0f * nf);
      z = nf / (2.0f * kPIf * theta * theta);
#pragma unroll
      for (int i = 0; i < 6; ++i) g[i] = z;
    } else {
      const int zs = solve_z_R_f<EDF, S::kScaled, false>(nf, ef, z, g);
      st |= zs;
      if (zs & ST_CLAMPED) theta = sqrtf(nf / (2.0f * kPIf * g[1]));
      else theta = 0.5f * g[1] / g[2] * ef / nf;
    }
    // conserved equilibrium moments from the double-float state: Z_1k from
    // n gamma, Z_2k from eps gamma^2 (a clamped BE state relaxes to its own
    // equilibrium energy 4 pi theta^3 g_3(z_c))
    const df2 ne = df_mul(df_join(F.n, F.eps), df_dup(F.gamma));
    const df nG = df_first(ne);
    df eG2 = df_mul(df_second(ne), F.gamma);
    if (st & ST_CLAMPED) eG2 = df_make(4.0f * kPIf * theta * theta * theta * g[2] * gf * gf, 0.0f);
    EqF q;
    dz_moments<EDF>(D, g, theta, uxf, uyf, gf, nG.hi, eG2.hi, q);
    // Z_20 = eps gamma^2 (1 + u^2/2), all in double-float
    const df dz10 = df_sub(nG, df_make(D.z1_hl[0], D.z1_hl[1]));
    const df dz20 = df_sub(df_add(eG2, df_mul(eG2, df_scale(F.u2, 0.5f))), df_make(D.z2_hl[0], D.z2_hl[1]));
    q.zr[1] = df_to_float(dz10);
    q.zr[3] = df_to_float(dz20);
    // Z_21 = (3/2) eps gamma^2 (u_x + i u_y) (Appendix; the rest state has none),
    // also from the double-float state rather than from FP32 eps gamma^2
    f2_split(df_to_float(df_mul(df_dup(df_mul(eG2, 1.5f)), F.u)), q.zr[4], q.zi[4]);
    remove_defects<EDF>(q);
    // constant tau, or the local tau = 4 (eta/s) / theta + 0.2546 of Sec. 3.5
    float itau = D.inv_tau_f;
    if (D.eta_s_f > 0.0f) itau = 1.0f / (4.0f * D.eta_s_f / theta + 0.2546f);
    float om[12];
    relax_rates(gf, uxf, uyf, itau, om);
    relax_cell<EDF, S, kImages || kHalo == 2>(D, q, om, col, fout + c);
  } else {
    for (int k = 0; k < kPairs; ++k)
      *reinterpret_cast<Pair<typename S::T>*>(fout + c + k * kSegW) = S::enc2(col[k * kThreads], D, 2 * (k % 3));
  }
  if (kImages || kHalo > 0)
    if (edge_warp) write_halo_mixed<EDF, S>(D, x, y, fout, col, ok, nf, uxf, uyf, gf, st, kImages);
  return st;
}

// Momentum weights (p_s, p_s^2) of the shells in work units.
struct PullW {
  f2 p[6];
};
template <int EDF, class S>
__device__ __forceinline__ PullW pull_weights(const DomDev& D) {
  PullW w;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    w.p[s] = f2_make(c_mt.p[EDF][s].x, c_mt.p[EDF][s].y);
    if constexpr (S::kScaled) w.p[s] = vmul(w.p[s], f2_dup(D.a_s[s]));
  }
  return w;
}
// (A_d, B_d) of a direction from its three pairs in work units, shell after shell
__device__ __forceinline__ f2 direction_sums(const f2 v[3], const PullW& w) {
  f2 ab = vmul(f2_dup(f2_lo(v[0])), w.p[0]);
  ab = vfma(f2_dup(f2_hi(v[0])), w.p[1], ab);
#pragma unroll
  for (int j = 1; j < 3; ++j) {
    ab = vfma(f2_dup(f2_lo(v[j])), w.p[2 * j], ab);
    ab = vfma(f2_dup(f2_hi(v[j])), w.p[2 * j + 1], ab);
  }
  return ab;
}

// Ask L2 for a tile's own blocks in rows y0-1 .. y0+kTileH of every plane: one
// contiguous segment per row, one bulk prefetch each.
template <class S>
__device__ __forceinline__ void prefetch_tile_l2(const DomDev& D, const Tile& tl, const typename S::T* fin) {
  const int r1 = min(tl.y0 + kTileH, D.ny);
  for (int r = tl.y0 - 1; r <= r1; ++r) {
    const typename S::T* p = fin + cell_rel(D, tl.x0, r);  // lane 0, plane 0 of the tile's block
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)),
                 "r"((unsigned)(kBlk * sizeof(typename S::T)))
                 : "memory");
  }
}

// One tile of the step (32 x 4 cells, or a packed ragged block): pull,
// collide, store (the thread's cell).
template <int EDF, class S, int kHalo>
__device__ __forceinline__ void step_tile_mixed(const StepArgs& a, int t, float* smf, int tid) {
  const Tile tl = a.tiles[t];
  const DomDev& D = a.doms[tl.dom];
  int x, y;
  if (!tile_cell(tl, threadIdx.x, threadIdx.y, x, y) || x >= D.nx || y >= D.ny) return;
  const typename S::T* __restrict__ fin = static_cast<const typename S::T*>(a.fin) + D.off;
  typename S::T* __restrict__ fout = static_cast<typename S::T*>(a.fout) + D.off;
#if RLBM_MIXED_L2_PREFETCH
  // (a packed tile uses at most half of each block it would fetch: not worth it)
  if (tid == 0 && tl.w == 0) prefetch_tile_l2<S>(D, tl, fin);
#endif
  const long long c = cell_rel(D, x, y);
  const Nbr nb = neighbours(D, x, y);
  // pull (FP32, work units) with the FP32 deviation moment sums
  f2 AB[12];
  f2* col = reinterpret_cast<f2*>(smf) + tid;
  const PullW w = pull_weights<EDF, S>(D);
#define RLBM_PULL_DIR(d)                                                                       \
  {                                                                                            \
    f2 v_[3];                                                                                  \
    _Pragma("unroll") for (int j = 0; j < 3; ++j) {                                            \
      v_[j] = S::work2(pull_pair<d, PullF32, S>(fin + c + (3 * d + j) * kSegW, nb), D, 2 * j); \
      col[(3 * d + j) * kThreads] = v_[j];                                                     \
    }                                                                                          \
    AB[d] = direction_sums(v_, w);                                                             \
  }
  RLBM_PULL_DIR(0) RLBM_PULL_DIR(1) RLBM_PULL_DIR(2) RLBM_PULL_DIR(3)
  RLBM_PULL_DIR(4) RLBM_PULL_DIR(5) RLBM_PULL_DIR(6) RLBM_PULL_DIR(7)
  RLBM_PULL_DIR(8) RLBM_PULL_DIR(9) RLBM_PULL_DIR(10) RLBM_PULL_DIR(11)
#undef RLBM_PULL_DIR
  const unsigned st = collide_mixed<EDF, S, false, kHalo>(D, x, y, c, AB, col, fout);
  if (st) atomicOr(a.status, st);
}

// kHalo = StepArgs::halo (see collide_mixed): 0 no halo writer, 0 and 1 no copy
// of the relaxed values into the column.
//
// Bound: HBM for the FP32 storages (2048^2 periodic, FP32 deviations: 376 us, 6.42
// TB/s of algorithmic traffic, 0.94 of the copy rate), instructions and the FP32 pipe
// for the 16-bit ones (328 us, 0.54 of it). Planes in pairs: one load or store moves
// the shells s, s + 1 of a direction, and the pull, the sums and the synthesis work on
// them as f32x2. With one plane per segment and scalar arithmetic the same step
// issued 1.6 times the instructions (2,774 per 32 cells, now 1,702): 461 us (FP32
// deviations), 500 us (BF16).
template <int EDF, class S, int kHalo>
__global__ void __launch_bounds__(kThreads, (mixed_min_blocks<S, kHalo>())) k_step_mixed(StepArgs a) {
  extern __shared__ float smf[];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
    step_tile_mixed<EDF, S, kHalo>(a, t, smf, tid);
  }
}

// ------------------------------------------- TMA-staged variant of the step
// Per 32 x 4 tile and direction d, one TMA box brings the three plane pairs of d
// for the tile's block of 32 cells and the blocks either side, rows y0-1 ..
// y0+kTileH, into shared memory (a box {64 elements, 3 pairs, 3 blocks, kTileH + 2 rows} of the
// 4D tensor {64, 36, nblk, ny + 2}); the bilinear pull reads its four
// neighbours there at fixed offsets (x - 1 of lane 0 and x + 1 of lane 31 in
// the neighbouring blocks). A ring of kStages boxes keeps the next directions --
// and, while a tile collides, the next tile's first directions -- in flight.
// The arithmetic is the same as k_step_mixed's, so the two variants give
// identical results.
template <class S>
struct TmaBox {
  using T = typename S::T;
  static constexpr int kBlock = kBoxPairs * kSegW;            // three pairs of one block
  static constexpr int kRow = kBoxBlocks * kBlock;            // three blocks of one row
  static constexpr unsigned kBytes = (unsigned)(kBoxElems * sizeof(T));
  static constexpr int kStageElems = kBoxElems;
};
constexpr int kStages = 3;  // ring depth in directions (a divisor of 12)

template <class S>
constexpr size_t tma_smem_bytes() {
  return kStages * (size_t)TmaBox<S>::kBytes + 72 * kThreads * sizeof(float) + kStages * sizeof(uint64_t);
}

// Issue the box of direction d of tile t into its ring stage (one thread).
template <class S>
__device__ __forceinline__ void tma_issue(const StepArgs& a, int t, int d, unsigned char* ring, uint64_t* bar) {
  const Tile tl = a.tiles[t];
  const void* map = static_cast<const unsigned char*>(a.tmaps) + (size_t)tl.dom * kTensorMapBytes;
  const int k = d % kStages;
  mbar_expect_tx(&bar[k], TmaBox<S>::kBytes);
  // elements from 0, pairs from 3d, blocks from the one left of the tile's
  // (x0 / 32 + 1 holds x0), rows from y = y0 - 1 (row index y0)
  tma_load_4d(ring + k * TmaBox<S>::kBytes, map, 0, 3 * d, tl.x0 / kBlkW, tl.y0, &bar[k]);
}

// Pull of direction d from its staged box; `cell` points at the cell's own
// value in shell 0 of that stage, oxm / oxp are the offsets of x - 1 / x + 1
// there (same weights and order of operations as pull_pair), col at the
// thread's shared-memory column.
template <int d, class S>
__device__ __forceinline__ f2 pull_dir_staged(const typename S::T* cell, int oxm, int oxp, const DomDev& D,
                                              const PullW& w, f2* col) {
  Nbr nb;
  nb.xm = oxm;
  nb.xp = oxp;
  nb.ym = -TmaBox<S>::kRow;
  nb.yp = TmaBox<S>::kRow;
  f2 v[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    v[j] = S::work2(pull_pair<d, PullF32, S>(cell + j * kSegW, nb), D, 2 * j);
    col[(3 * d + j) * kThreads] = v[j];
  }
  return direction_sums(v, w);
}

template <int EDF, class S>
__global__ void __launch_bounds__(kThreads, 512 / kThreads) k_step_mixed_tma(StepArgs a) {
  using T = typename S::T;
  using TB = TmaBox<S>;
  extern __shared__ __align__(128) unsigned char smt[];
  unsigned char* ring = smt;
  float* smf = reinterpret_cast<float*>(smt + kStages * TB::kBytes);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smt + kStages * TB::kBytes + 72 * kThreads * sizeof(float));
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  if (blockIdx.x >= a.ntiles) return;  // whole block
  const unsigned long long wait_ns = a.wait_ns ? a.wait_ns : kDefaultWaitNs;
  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < kStages; ++k) mbar_init(&bar[k], 1);
    fence_barrier_init();
  }
  __syncthreads();
  // thread 0 tracks the loads in flight per stage (for the drain on a timeout)
  unsigned inflight = 0, issued[kStages] = {};
  if (tid == 0) {
#pragma unroll
    for (int d = 0; d < kStages; ++d) {
      tma_issue<S>(a, blockIdx.x, d, ring, bar);
      inflight |= 1u << d;
      ++issued[d];
    }
  }
  // the cell's own value in shell 0 of stage 0 (row ty + 1, middle block, lane
  // tx), the offsets of its x neighbours, and its column
  const T* cell0 = reinterpret_cast<const T*>(ring) + (threadIdx.y + 1) * TB::kRow + TB::kBlock + 2 * threadIdx.x;
  const int oxm = threadIdx.x > 0 ? -2 : -TB::kBlock + 2 * (kBlkW - 1);
  const int oxp = threadIdx.x < kBlkW - 1 ? 2 : TB::kBlock - 2 * (kBlkW - 1);
  f2* col = reinterpret_cast<f2*>(smf) + tid;
  unsigned it = 0;  // tiles done by this block: stage uses so far = it * 12 / kStages + d / kStages
  for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++it) {
    const Tile tl = a.tiles[t];
    const DomDev& D = a.doms[tl.dom];
    const int x = tl.x0 + threadIdx.x, y = tl.y0 + threadIdx.y;
    const int tnext = t + gridDim.x;
    const unsigned use0 = it * (12 / kStages);
    const PullW w = pull_weights<EDF, S>(D);
    f2 AB[12];
    // every lane pulls (lanes outside the domain read the box's padding and
    // fill only their own column, which is never stored)
#define RLBM_STAGED_DIR(d)                                                                      \
  {                                                                                             \
    constexpr int k_ = (d) % kStages;                                                           \
    const bool ok_ = mbar_wait(&bar[k_], (use0 + (d) / kStages) & 1, wait_ns);                  \
    AB[d] = pull_dir_staged<d, S>(cell0 + k_ * TB::kStageElems, oxm, oxp, D, w, col);           \
    if (__syncthreads_or(!ok_)) goto timed_out;                                                 \
    if (tid == 0) {                                                                             \
      inflight &= ~(1u << k_);                                                                  \
      const int tt_ = (d) + kStages < 12 ? t : tnext;                                           \
      if (tt_ < a.ntiles) {                                                                     \
        tma_issue<S>(a, tt_, ((d) + kStages) % 12, ring, bar);                                  \
        inflight |= 1u << k_;                                                                   \
        ++issued[k_];                                                                           \
      }                                                                                         \
    }                                                                                           \
  }
    RLBM_STAGED_DIR(0) RLBM_STAGED_DIR(1) RLBM_STAGED_DIR(2) RLBM_STAGED_DIR(3)
    RLBM_STAGED_DIR(4) RLBM_STAGED_DIR(5) RLBM_STAGED_DIR(6) RLBM_STAGED_DIR(7)
    RLBM_STAGED_DIR(8) RLBM_STAGED_DIR(9) RLBM_STAGED_DIR(10) RLBM_STAGED_DIR(11)
#undef RLBM_STAGED_DIR
    if (x < D.nx && y < D.ny) {
      T* __restrict__ fout = static_cast<T*>(a.fout) + D.off;
      const unsigned st = collide_mixed<EDF, S, true>(D, x, y, cell_rel(D, x, y), AB, col, fout);
      if (st) atomicOr(a.status, st);
    }
  }
  return;
timed_out:
  // a copy did not land in time: report it, let the copies still in flight
  // finish (bounded by the default limit, whatever the limit of the waits
  // above) so that none writes shared memory after exit, return
  if (tid == 0) {
    atomicOr(a.status, ST_TIMEOUT);
#pragma unroll
    for (int k = 0; k < kStages; ++k)
      if (inflight & (1u << k)) mbar_wait(&bar[k], (issued[k] - 1) & 1);
  }
}

// Macroscopic fields (n, theta, ux, uy, z) of a mixed storage's populations in
// the collision's own arithmetic -- the FP32 pull and deviation sums, the
// double-float totals and Landau frame (Eqs. 20-25), the FP32 fugacity solve --
// written as FP64 (the double-float values to nearest). It runs on the FP32 pipe, the
// conversions included (df_to_f64; on the FP64 unit they were a third of its time);
// the FP64 read-out k_fields, at 1/64 of that rate, serves the diagnostics. Bound: HBM.
template <int EDF, class S>
__global__ void __launch_bounds__(kThreads) k_fields_mixed(FieldsArgs a) {
  int dom, x, y;
  cell_of_launch(a.tiles, a.dom, dom, x, y);
  const DomDev& D = a.doms[dom];
  if (x >= D.nx || y >= D.ny) return;
  const typename S::T* __restrict__ f = static_cast<const typename S::T*>(a.f) + D.off;
  const long long c = cell_rel(D, x, y);
  if (a.tiles && threadIdx.x == 0 && threadIdx.y == 0) prefetch_tile_l2<S>(D, a.tiles[blockIdx.x], f);
  f2 AB[12];
  {
    const PullW w = pull_weights<EDF, S>(D);
    const Nbr nb = neighbours(D, x, y);
    const bool streamed = a.streamed != 0;
#define RLBM_FIELDS_DIR(d)                                                                          \
  {                                                                                                 \
    f2 v_[3];                                                                                       \
    _Pragma("unroll") for (int j = 0; j < 3; ++j) {                                                 \
      const typename S::T* pl = f + c + (3 * d + j) * kSegW;                                        \
      const f2 r = streamed ? pull_pair<d, PullF32, S>(pl, nb)                                      \
                            : S::raw2(*reinterpret_cast<const Pair<typename S::T>*>(pl));           \
      v_[j] = S::work2(r, D, 2 * j);                                                                \
    }                                                                                               \
    AB[d] = direction_sums(v_, w);                                                                  \
  }
    RLBM_FIELDS_DIR(0) RLBM_FIELDS_DIR(1) RLBM_FIELDS_DIR(2) RLBM_FIELDS_DIR(3)
    RLBM_FIELDS_DIR(4) RLBM_FIELDS_DIR(5) RLBM_FIELDS_DIR(6) RLBM_FIELDS_DIR(7)
    RLBM_FIELDS_DIR(8) RLBM_FIELDS_DIR(9) RLBM_FIELDS_DIR(10) RLBM_FIELDS_DIR(11)
#undef RLBM_FIELDS_DIR
  }
  FrameDf F;
  unsigned st = landau_df(moments_df(D, AB), F);
  double on = nan(""), oth = nan(""), oux = nan(""), ouy = nan(""), oz = nan("");
  if (!(st & ST_NONPHYSICAL)) {
    const float nf = df_to_float(F.n), ef = df_to_float(F.eps);
    float theta, z, g[6];
    if (EDF == EDF_MJ) {
      theta = ef / (2.0f * nf);
      z = nf / (2.0f * kPIf * theta * theta);
    } else {
      const int zs = solve_z_R_f<EDF, S::kScaled, true>(nf, ef, z, g);
      st |= zs;
      if (zs & ST_CLAMPED) theta = sqrtf(nf / (2.0f * kPIf * g[1]));
      else theta = 0.5f * g[1] / g[2] * ef / nf;
    }
    const df ux = df_first(F.u), uy = df_second(F.u);
    on = df_to_f64(F.n);
    oux = df_to_f64(ux);
    ouy = df_to_f64(uy);
    oth = f32_to_f64(theta);
    oz = f32_to_f64(z);
  }
  const long long i = (a.tiles ? D.foff : 0) + (long long)y * D.nx + x;
  if (a.n) a.n[i] = on;
  if (a.theta) a.theta[i] = oth;
  if (a.ux) a.ux[i] = oux;
  if (a.uy) a.uy[i] = ouy;
  if (a.z) a.z[i] = oz;
  if (st) atomicOr(a.status, st);
}

// The mixed storages' read-out: the fields in the collision's arithmetic, or
// the FP64 kernel when diagnostics are asked for.
template <class S>
cudaError_t launch_fields_mixed_t(int edf, const FieldsArgs& a, int nx, int ny, cudaStream_t s) {
  if (a.diag) return launch_fields_t<S>(edf, a, nx, ny, s);
  const dim3 grid = launch_grid(a.tiles, a.ntiles, nx, ny);
  switch (edf) {
    case EDF_MJ: k_fields_mixed<EDF_MJ, S><<<grid, dim3(kTileW, kTileH), 0, s>>>(a); break;
    case EDF_FD: k_fields_mixed<EDF_FD, S><<<grid, dim3(kTileW, kTileH), 0, s>>>(a); break;
    default: k_fields_mixed<EDF_BE, S><<<grid, dim3(kTileW, kTileH), 0, s>>>(a); break;
  }
  return cudaGetLastError();
}

// f = f^eq of the given fields in a mixed storage (time zero), halo included:
// the collision's FP32 equilibrium deviations (dz_moments, dfeq_pair, with the
// tables' conserved-moment defects removed) from the FP64 input fields. Its
// rounding is that of every collision of the mixed step, and it runs on the
// FP32 pipe (an FP64 initialiser costs as much as ten mixed steps on GB300).
template <int EDF, class S>
__global__ void __launch_bounds__(kThreads) k_init_mixed(InitArgs a) {
  extern __shared__ float smi[];
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  int dom, x, y;
  cell_of_launch(a.tiles, a.dom, dom, x, y);
  const DomDev& D = a.doms[dom];
  if (x >= D.nx || y >= D.ny) return;
  const long long i = (a.tiles ? D.foff : 0) + (long long)y * D.nx + x;
  const float theta = (float)a.theta[i], ux = (float)a.ux[i], uy = (float)a.uy[i];
  unsigned st = 0;
  float z, n, g[6];
  if (a.kind == 1) {
    z = (float)a.a[i];
    g_allf<EDF>(z, g);
    n = 2.0f * kPIf * theta * theta * g[1];
  } else {
    n = (float)a.a[i];
    st |= (theta > 0.0f && n > 0.0f) ? solve_z_nt_f<EDF, S::kScaled, true>(n, theta, z, g) : 0;
  }
  const float u2 = fmaf(ux, ux, __fmul_rn(uy, uy));
  const bool ok = (u2 < 1.0f) && (theta > 0.0f) && (n > 0.0f) && isfinite(z) && isfinite(u2);
  if (!ok) st |= ST_NONPHYSICAL;
  const float gam = ok ? 1.0f / sqrtf(1.0f - u2) : 1.0f;
  typename S::T* __restrict__ f = static_cast<typename S::T*>(a.f) + D.off;
  const long long c = cell_rel(D, x, y);
  f2* col = reinterpret_cast<f2*>(smi) + tid;
  using P = Pair<typename S::T>;
  // only warps with a cell on the domain's edge have halo cells to write
  const bool edge_warp = __any_sync(__activemask(), x == 0 || x == D.nx - 1 || y == 0 || y == D.ny - 1);
  if (ok) {
    EqF q;
    dz_moments<EDF>(D, g, theta, ux, uy, gam, -1.0f, -1.0f, q);
    remove_defects<EDF>(q);
#pragma unroll 1
    for (int j = 0; j < 3; ++j) {
      f2 fe[12];
      dfeq_work<EDF, S>(D, j, q, fe);
#pragma unroll
      for (int d = 0; d < 12; ++d) {
        col[(3 * d + j) * kThreads] = fe[d];
        *reinterpret_cast<P*>(f + c + (3 * d + j) * kSegW) = S::enc2(fe[d], D, 2 * j);
      }
    }
  } else {
    for (int k = 0; k < kPairs; ++k) {
      col[k * kThreads] = f2_dup(__int_as_float(0x7fc00000));  // NaN
      *reinterpret_cast<P*>(f + c + k * kSegW) = S::enc2(col[k * kThreads], D, 2 * (k % 3));
    }
  }
  if (edge_warp) write_halo_mixed<EDF, S>(D, x, y, f, col, ok, n, ux, uy, gam, st, true);
  if (st) atomicOr(a.status, st);
}

template <class S>
cudaError_t launch_init_mixed_t(int edf, const InitArgs& a, int nx, int ny, cudaStream_t s) {
  const dim3 grid = launch_grid(a.tiles, a.ntiles, nx, ny);
  switch (edf) {
    case EDF_MJ: k_init_mixed<EDF_MJ, S><<<grid, dim3(kTileW, kTileH), kSmemF, s>>>(a); break;
    case EDF_FD: k_init_mixed<EDF_FD, S><<<grid, dim3(kTileW, kTileH), kSmemF, s>>>(a); break;
    default: k_init_mixed<EDF_BE, S><<<grid, dim3(kTileW, kTileH), kSmemF, s>>>(a); break;
  }
  return cudaGetLastError();
}

// Reference rest equilibrium of every domain (FP64), its FP32 rounding and
// the reference moments, written into the device descriptors.
template <int EDF>
__global__ void k_prepare_refs(DomDev* doms, int ndom) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ndom) return;
  DomDev& D = doms[i];
  double z, g[6];
  solve_z_from_n_theta<EDF, false>(D.ref_n, D.ref_theta, z, g);
  double fact = 1.0, th = D.ref_theta, thp = th;
  for (int n = 0; n < 6; ++n) {
    if (n > 0) { fact *= n; thp *= th; }
    D.zref[n] = 2.0 * PI * fact * g[n] * thp * c_pnk[3 * (n * (n + 1) / 2)];
  }
  double n0 = 0.0, t00 = 0.0;
  for (int s = 0; s < 6; ++s) {
    double fe = 0.0;
    for (int n = 0; n < 6; ++n) fe += c_Q[kOrder5][EDF][qoff(0) + s * 6 + n] * D.zref[n];
    const float ff = (float)fe;
    D.fref[s] = ff;
    D.rres[s] = (float)(fe - (double)ff);
    const float as = (float)((double)ff * D.scale);
    D.a_s[s] = as;
    D.b_s[s] = 1.0f / as;
    n0 += 12.0 * (double)ff * c_p[EDF][s];
    t00 += 12.0 * (double)ff * c_p2[EDF][s];
  }
  D.n0ref = n0;
  D.t00ref = t00;
  double r1 = 0.0, r2 = 0.0;
  for (int s = 0; s < 6; ++s) {
    r1 += 12.0 * (double)D.rres[s] * (double)c_mt.p[EDF][s].x;
    r2 += 12.0 * (double)D.rres[s] * (double)c_mt.p[EDF][s].y;
  }
  D.zeff1 = n0 + r1;
  D.zeff2 = t00 + r2;
  const double v4[4] = {D.n0ref, D.t00ref, D.zeff1, D.zeff2};
  float* pairs[4] = {D.n0_hl, D.t00_hl, D.z1_hl, D.z2_hl};
  for (int k = 0; k < 4; ++k) {
    pairs[k][0] = (float)v4[k];
    pairs[k][1] = (float)(v4[k] - (double)pairs[k][0]);
  }
  for (int n = 0; n < 6; ++n) D.zref_f[n] = (float)D.zref[n];
}

// ------------------------------------------------------------- launchers
template <class S, int EDF>
static cudaError_t prepare_tma_t() {
  cudaError_t e = cudaFuncSetAttribute(k_step_mixed_tma<EDF, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)tma_smem_bytes<S>());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_step_mixed_tma<EDF, S>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}

template <class S, int EDF>
static cudaError_t prepare_mixed_t() {
  cudaError_t e = cudaFuncSetAttribute(k_init_mixed<EDF, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_step_mixed<EDF, S, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_step_mixed<EDF, S, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_step_mixed<EDF, S, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF);
}

// Shared-memory limits of a storage's kernels.
template <class S>
static cudaError_t prepare_s() {
  cudaError_t e;
  if ((e = prepare_mixed_t<S, EDF_MJ>())) return e;
  if ((e = prepare_mixed_t<S, EDF_FD>())) return e;
  if ((e = prepare_mixed_t<S, EDF_BE>())) return e;
  if ((e = prepare_tma_t<S, EDF_MJ>())) return e;
  if ((e = prepare_tma_t<S, EDF_FD>())) return e;
  if ((e = prepare_tma_t<S, EDF_BE>())) return e;
  if ((e = prepare_common_t<S, EDF_MJ>())) return e;
  if ((e = prepare_common_t<S, EDF_FD>())) return e;
  return prepare_common_t<S, EDF_BE>();
}

template <class S>
static cudaError_t step_s(int edf, const StepArgs& a, int grid, cudaStream_t s) {
  if (a.tmaps) {  // TMA-staged variant; without descriptors the pull goes through L1
    const size_t sm = tma_smem_bytes<S>();
    switch (edf) {
      case EDF_MJ: k_step_mixed_tma<EDF_MJ, S><<<grid, dim3(kTileW, kTileH), sm, s>>>(a); break;
      case EDF_FD: k_step_mixed_tma<EDF_FD, S><<<grid, dim3(kTileW, kTileH), sm, s>>>(a); break;
      default: k_step_mixed_tma<EDF_BE, S><<<grid, dim3(kTileW, kTileH), sm, s>>>(a); break;
    }
    return cudaGetLastError();
  }
  const dim3 blk(kTileW, kTileH);
#define RLBM_STEP_L1(H)                                                           \
  switch (edf) {                                                                  \
    case EDF_MJ: k_step_mixed<EDF_MJ, S, H><<<grid, blk, kSmemF, s>>>(a); break; \
    case EDF_FD: k_step_mixed<EDF_FD, S, H><<<grid, blk, kSmemF, s>>>(a); break; \
    default: k_step_mixed<EDF_BE, S, H><<<grid, blk, kSmemF, s>>>(a); break;     \
  }
  if (a.halo == 0) {
    RLBM_STEP_L1(0)
  } else if (a.halo == 1) {
    RLBM_STEP_L1(1)
  } else {
    RLBM_STEP_L1(2)
  }
#undef RLBM_STEP_L1
  return cudaGetLastError();
}

// The launchers of one storage format, exported by its translation unit.
struct MixedUnit {
  cudaError_t (*prepare)();
  cudaError_t (*step)(int edf, const StepArgs& a, int grid, cudaStream_t s);
  cudaError_t (*init)(int edf, const InitArgs& a, int nx, int ny, cudaStream_t s);
  cudaError_t (*fields)(int edf, const FieldsArgs& a, int nx, int ny, cudaStream_t s);
  cudaError_t (*copy)(const CopyArgs& a, cudaStream_t s);
};

template <class S>
constexpr MixedUnit mixed_unit() {
  return MixedUnit{&prepare_s<S>, &step_s<S>, &launch_init_mixed_t<S>, &launch_fields_mixed_t<S>,
                   &launch_copy_t<S>};
}

extern const MixedUnit kMixedF32, kMixedF32Dev, kMixedBF16, kMixedF16;

}  // namespace rlbm
