// Per-nucleus (or per-point) device helpers of the FP64 path's nucleus loop (step S2), shared by the coupling kernel and
// the electrostatic potential: the scaled harmonic columns in fixed point, the Boys values and radial factors, and
// their constants.  Each translation unit that includes this header has its own copy of the constants and uploads them
// with upload_nucleus_constants().
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "shgo_fixed.cuh"
#include "shgo_internal.h"
#include "shgo_math.h"

namespace shgo {
namespace {

constexpr int kCS = 33;  // columns of a table row: 32 and one, so that 8-byte loads of different rows differ in bank
constexpr double kMagic = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer in the low word

__constant__ BoysConst k_boys;
// Step l -> l + 1 of column m (l >= m >= 0), at l (l + 1) / 2 + m: V = 2^e U obeys
// V_{l+1} = 2^a z V_l + n V_{l-1}; (n's limbs, a, e(l, m)).  Two sets of scales: e_0 for x, y as they are (|V| <= 1 as
// 2^e_0 <= N_lm and |S_lm| <= 1), e_1 for a chunk close to the axis, whose x, y are scaled up to the order of 1
// (2^e_1 <= 1 / max |V / (x + iy)^m|, reached at z = 1).
constexpr int kSteps = (kLamDer + 1) * (kLamDer + 2) / 2;
__constant__ int4 k_step[2 * kSteps];
__device__ int4 g_step[2 * kSteps];  // the same, for copies to shared memory
// Per set and harmonic row h = (L, M): |M| | e(L, M) << 8 | L << 16.
constexpr int kRows = (kLamDer + 1) * (kLamDer + 1);
__device__ int g_row[2 * kRows];
// a_{L,k} = sqrt(pi)/2 sum_{j<=k} (2(L+j)-1)!! / (2^{L+j} j!) at L (kLamDer / 2 + 1) + k, and 2 pi k!.
__device__ double g_far[(kLamDer + 1) * (kLamDer / 2 + 1)];
__device__ double g_kfact[kLamDer / 2 + 1];

// T from which F_n(T), n <= Lambda, is asymptotic: Q(Lambda + 1/2, T) = 2^-56 (the regularised upper incomplete
// gamma function is the relative deviation), rounded up; inside the grid (80) for every order.
__host__ __device__ constexpr double far_t(int lam) {
  constexpr double t[kLamDer + 1] = {36.5, 40.9, 44.3, 47.4, 50.2, 52.8, 55.4, 57.8, 60.2,
                                     62.5, 64.7, 66.9, 69.0, 71.1, 73.1, 75.2, 77.2, 79.1};
  return t[lam];
}

__host__ __device__ constexpr int beta_first(int lam, int L) {  // first radial row of L
  int n = 0;
  for (int l = 0; l < L; ++l) n += ((lam - l) >> 1) + 1;
  return n;
}

// C - A of a nucleus (or point) at c in the pair frame Q.
__device__ __forceinline__ void frame_coords(const double* Q, const double* xa, const double* c, double& x, double& y,
                                             double& z) {
  const double vx = c[0] - xa[0], vy = c[1] - xa[1], vz = c[2] - xa[2];
  x = Q[0] * vx + Q[1] * vy + Q[2] * vz;
  y = Q[3] * vx + Q[4] * vy + Q[5] * vz;
  z = Q[6] * vx + Q[7] * vy + Q[8] * vz;
}
// High word of the least |d|^2 that counts as nonzero: |d| below 2^-500 counts as 0, only L = 0 survives there.
constexpr int kTinyHi = 0x01700000;

// 2^a z v + n w (fixed point; the caller passes z's limbs already shifted by a).
__device__ __forceinline__ fx fx_step(fx z, fx v, int nh, int nl, fx w) {
  long long hh = fx_mad(z.h, v.h, 0), mid = fx_mad(z.h, v.l, 0);
  mid = fx_mad(z.l, v.h, mid);
  hh = fx_mad(nh, w.h, hh);
  mid = fx_mad(nh, w.l, mid);
  mid = fx_mad(nl, w.h, mid);
  return fx_split(fx_sum(hh, mid));
}

// Columns m = +-am, am in [A0, A1), of V_lm into rows h of St at column c.
template <int LAM>
__device__ __forceinline__ void harmonic_columns(int A0, int A1, int set, fx x, fx y, fx z, int2* St, int c) {
  fx dp = {1 << kFxLimb, 0}, dm = {0, 0};  // (x + iy)^am
  const fx ny = fx_neg(y);
#pragma unroll 1
  for (int am = 0; am < A1; ++am) {
    if (am >= A0) {
      fx p0 = {0, 0}, p1 = dp, m0 = {0, 0}, m1 = dm;
#pragma unroll 1
      for (int l = am;; ++l) {
        const int h = l * l + l;
        St[(h + am) * kCS + c] = make_int2(p1.h, p1.l);
        if (am) St[(h - am) * kCS + c] = make_int2(m1.h, m1.l);
        if (l == LAM) break;
        const int4 s = k_step[set + l * (l + 1) / 2 + am];
        const fx za = {z.h << s.z, z.l << s.z};
        const fx pn = fx_step(za, p1, s.x, s.y, p0);
        p0 = p1;
        p1 = pn;
        if (am) {
          const fx mn = fx_step(za, m1, s.x, s.y, m0);
          m0 = m1;
          m1 = mn;
        }
      }
    }
    const fx t = fx_step(x, dp, ny.h, ny.l, dm);
    dm = fx_step(y, dp, x.h, x.l, dm);
    dp = t;
  }
}

// G_n, n = 0..LAM.  near: G_n = Z t^n F_n(T), t = sqrt(T), from the Taylor expansion of F_LAM about the nearest grid
// point and the downward recursion F_n = (2T F_{n+1} + exp(-T)) / (2n + 1) in scaled form, and tau_k = t^k / k!;
// otherwise the far form G_n = Z v^{n+1}, v = 1/t.  top: the Boys grid of order LAM.
template <int LAM>
__device__ __forceinline__ void radial_factors(bool near, double T, double t, double v, double Z,
                                               const double2* __restrict__ top, double (&G)[LAM + 1],
                                               double (&tau)[LAM / 2 + 1]) {
#pragma unroll
  for (int k = 0; k <= LAM / 2; ++k) tau[k] = 0.0;
  if (near) {
    const double tm = fma(T, kBoysInvH, kMagic);
    const int g = min(max(__double2loint(tm), 0), kBoysTopRows - 1);
    const double dT = fma(tm - kMagic, 1.0 / kBoysInvH, -T);  // T_g - T
    const double2* row = top + (size_t)g * (kBoysTopStride / 2);
    double f, ew = 1.0;
    {
      const double2 r3 = __ldg(row + 3), r2 = __ldg(row + 2), r1 = __ldg(row + 1), r0 = __ldg(row);
      f = fma(r3.y, dT, r3.x);
      f = fma(f, dT, r2.y);
      f = fma(f, dT, r2.x);
      f = fma(f, dT, r1.y);
      f = fma(f, dT, r1.x);
      f = fma(f, dT, r0.y);
      f = fma(f, dT, r0.x);
    }
    if constexpr (LAM > 0) {
      ew = 1.0 / 5040.0;
      ew = fma(ew, dT, 1.0 / 720.0);
      ew = fma(ew, dT, 1.0 / 120.0);
      ew = fma(ew, dT, 1.0 / 24.0);
      ew = fma(ew, dT, 1.0 / 6.0);
      ew = fma(ew, dT, 0.5);
      ew = fma(ew, dT, 1.0);
      ew = fma(ew, dT, 1.0);
    }
    double zt = Z, tp = t;  // Z t^Lambda by squaring
#pragma unroll
    for (int bit = 0; (1 << bit) <= LAM; ++bit) {
      if ((LAM >> bit) & 1) zt *= tp;
      if ((2 << bit) <= LAM) tp *= tp;
    }
    G[LAM] = zt * f;
    if constexpr (LAM > 0) {
      // F_n = (2T F_{n+1} + exp(-T)) / (2n + 1), scaled: G_n = (2t G_{n+1} + Z t^n exp(-T)) / (2n + 1)
      G[0] = Z * (__ldg(row + 4).x * ew);
#pragma unroll
      for (int n = 1; n < LAM; ++n) G[n] = G[n - 1] * t;
      const double t2 = t + t;
#pragma unroll
      for (int n = LAM - 1; n >= 0; --n) G[n] = fma(t2, G[n + 1], G[n]) * k_boys.inv_odd[n];
      tau[0] = 1.0;
#pragma unroll
      for (int k = 1; k <= LAM / 2; ++k) tau[k] = tau[k - 1] * (t * k_boys.inv_int[k]);
    }
  } else {
    G[0] = Z * v;
#pragma unroll
    for (int n = 1; n <= LAM; ++n) G[n] = G[n - 1] * v;
  }
}

inline cudaError_t upload_nucleus_constants() {
  const HarmCoef& hc = harm_coef_host();
  std::vector<int4> step(2 * kSteps);
  std::vector<int> row(2 * kRows);
  for (int set = 0; set < 2; ++set) {
    // e(l, m): the largest exponent within the set's bound that grows by at most one from l to l + 1
    int ex[kLamDer + 1][kLamDer + 1] = {};
    for (int m = 0; m <= kLamDer; ++m) {
      double q0 = 0.0, q1 = 1.0;  // V / (x + iy)^m at z = 1, unscaled
      for (int l = m; l <= kLamDer; ++l) {
        const double bound = set == 0 ? hc.n[harm_index(l, m)] : 1.0 / q1;
        int e = 0;
        while (std::ldexp(1.0, e + 1) <= bound) ++e;
        ex[l][m] = l > m ? std::min(e, ex[l - 1][m] + 1) : 0;
        const double q2 = q1 - (l > m ? (double)(l * l - m * m) / (4 * l * l - 1) : 0.0) * q0;
        q0 = q1;
        q1 = q2;
      }
    }
    for (int l = 0; l <= kLamDer; ++l)
      for (int m = 0; m <= l; ++m) {
        int4 s = make_int4(0, 0, 0, ex[l][m]);
        if (l < kLamDer) s.z = ex[l + 1][m] - ex[l][m];
        if (l > m && l < kLamDer) {
          // -gamma_lm 2^(e(l+1) - e(l-1)) = -(l^2 - m^2) / (4 l^2 - 1) 2^(..), rounded to 2^-58
          const __int128 num = (__int128)(l * l - m * m) << (kFxBits + ex[l + 1][m] - ex[l - 1][m]);
          const long long den = 4 * l * l - 1, qq = -(long long)((2 * num + den) / (2 * den));
          const long long lo = (long long)((unsigned long long)qq << (64 - kFxLimb)) >> (64 - kFxLimb);
          s.x = (int)((qq - lo) >> kFxLimb);
          s.y = (int)lo;
        }
        step[set * kSteps + l * (l + 1) / 2 + m] = s;
        row[set * kRows + harm_index(l, m)] = row[set * kRows + harm_index(l, -m)] = m | ex[l][m] << 8 | l << 16;
      }
  }
  double far[(kLamDer + 1) * (kLamDer / 2 + 1)] = {}, kf[kLamDer / 2 + 1];
  for (int L = 0; L <= kLamDer; ++L) {
    long double g = 0.886226925452758013649083741670572591398L, s = 0.0L, jf = 1.0L;  // Gamma(L + j + 1/2) / 2
    for (int n = 1; n <= L; ++n) g *= (2 * n - 1) / 2.0L;
    for (int k = 0; k <= kLamDer / 2; ++k) {
      s += g / jf;
      far[L * (kLamDer / 2 + 1) + k] = (double)s;
      g *= (2 * (L + k) + 1) / 2.0L;
      jf *= k + 1;
    }
  }
  kf[0] = 6.283185307179586476925286766559;
  for (int k = 1; k <= kLamDer / 2; ++k) kf[k] = kf[k - 1] * k;
  cudaError_t e = cudaMemcpyToSymbol(k_boys, &boys_const_host(), sizeof(BoysConst));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(k_step, step.data(), sizeof(int4) * step.size());
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_step, step.data(), sizeof(int4) * step.size());
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_row, row.data(), sizeof(int) * row.size());
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_far, far, sizeof(far));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_kfact, kf, sizeof(kf));
  return e;
}

}  // namespace
}  // namespace shgo
