// FP64 coupling kernel (step S2), one instantiation per Lambda = la + lb (and la + lb + 1 for derivatives).
//
// For one primitive pair and its nuclei C, in the pair frame with d = C - P:
//   R'[L,M,k] = 2 pi k! p^{-(k+1)} sum_C Z_C S_LM(d) beta_{L,k}(T) / k!,
//   beta_{L,k} / k! = sum_{j<=k} T^j / j! F_{L+j}(T),  T = p |d|^2,
// the radial part of the corrected one-centre integral (Eq. 12 with the same-centre coupling restored) before the
// Clebsch-Gordan coupling of the pair kernel.  With t = sqrt(T), u = d/|d| and S_LM(u) = N_LM U_LM(u),
//   S_LM(d) beta_{L,k} / k! = p^{-L/2} N_LM U_LM(u) b_{L,k},   b_{L,k} = sum_{j<=k} t^j / j! (t^{L+j} F_{L+j}).
//
// What bounds it: FP64 issues 1.7 lanes per clock and SM on GB300, integer multiply-adds 62 (measured).  So FP64 is kept for
// what needs its range (geometry, Boys values, radial sums), once per nucleus, and the rest, the harmonics and the
// sums over nuclei, runs in 58-bit fixed point (shgo_fixed.cuh), which has more bits than an FP64 mantissa at full scale.
//
// The nuclei of a chunk of 32 fall in three kinds, and take columns of the shared tables in this order:
//  - near: T below kFarT[Lambda].  Boys values by Taylor expansion from a grid that reaches that T (one branch, no
//    asymptotic form), radial sums b_{L,k}, one table row per (L, k).
//  - far: F_n(T) equals its asymptotic form (2n-1)!!/2^n sqrt(pi)/2 T^{-n-1/2} to 2^-56, so T^j F_{L+j} does not depend
//    on j but by a constant: b_{L,k} = a_{L,k} t^{-(L+1)}, and one sum per (L, M) serves every k.  In a molecule most
//    nuclei are far (T = 40 is 3.6 bohr at p = 3): no Boys values, Lambda + 1 radial values instead of one per (L, k),
//    (Lambda + 1)^2 sums instead of C(Lambda + 3, 3).
//  - axis: on the line through A and B, as the nuclei of A and B themselves.  U_LM vanishes there but for M = 0, and
//    these nuclei dominate the radial values, so they would set the scale of sums they have no part in: they are
//    added in FP64 to the M = 0 entries alone.
// Radial rows are scaled by the largest exponent among the row's columns, near and far separately; harmonic rows by a
// power of two per (l, |m|), and x, y of a chunk close to the axis by that of the chunk's largest.  A sum is therefore within
// 32 x 2^-59 or so of its scale, the row's largest radial value times the harmonics' bound, where an FP64 sum rounds at
// 2^-53 of its partial sums: entries (L, M) much smaller than their row (x or y of every nucleus far below that of one that
// sets the scale) have fewer digits of their own than in FP64, the block's larger elements have more.
//
// Phases of a block (NW warps, one primitive pair at a time): warp 0, lane = nucleus: geometry, kinds, radial rows;
// all warps: the radial rows into fixed point, then for 16 columns at a time (a smaller table, so more blocks on an SM) the
// harmonics, |m| split over the warps by cost and the two signs of m on the halves of a warp; thread = (L, M): sums over
// the far columns; thread = R' entry: sums over the near columns, far part, axis part and scales.
//
// Measured (GB300, whole calls, against the same kernel with every step in FP64): V of 32 atoms with l <= 6 501 -> 404 us,
// of a contracted 29-atom molecule 7.00 -> 4.40 ms, of six such molecules in a batch 53.1 -> 29.8 ms; dV/dA of the
// 32 atoms 1.63 -> 1.50 ms.  Tables of 32 columns to 16, rows converted by all warps, coordinates kept over a shell pair's
// primitive pairs (after the pair kernel's contraction): 3.79 -> 3.69 ms, batch 27.6 -> 25.2 ms.  Errors against 64-bit
// quadrature are the same to two digits.  At Lambda <= 2 the FP64 pipe is 76 % busy (84 % is what plain DFMAs reach), from
// Lambda 4 on a primitive pair's dependent chains bound it (15 to 20 warps on an SM, FP64 pipe 45 to 55 % busy).
// Small calls, where a launch is one chain (7 to 9 us at Lambda <= 4): block tables by asynchronous copies, harmonic steps and row
// codes in shared memory, shorter sums: V of 14 atoms with l <= 2 43 -> 42 us, of 4 contracted atoms 46 -> 45, of 3 atoms
// with l <= 2 33.3 -> 33.0 (all in FP64: 45, 57, 31.5); large calls 1 to 2 % (29-atom molecule 3.64 -> 3.57 ms).  One preferred
// split of shared memory for all kernels of a call saves 3 to 7 us of device time there, but setting it costs a quarter of a
// microsecond of host time per launch, and calls on changing buffers are bound by the host: 57 -> 60 us.
#include <cuda_runtime.h>

#include <utility>
#include <vector>

#include "shgo_internal.h"
#include "shgo_nucleus.cuh"

namespace shgo {

namespace {

constexpr int kNch = 32;        // nuclei per chunk
// Boys grid per top order Lambda: row g holds F_{Lambda+k}(T_g) / k!, k = 0..7, exp(-T_g), 0.
__device__ double2 g_boys_top[(kLamDer + 1) * kBoysTopRows * kBoysTopStride / 2];

// Warps per block: one where a warp's tables leave an SM full of blocks, more where the harmonic columns are many and
// the tables large (the warps of a block share them).
__host__ __device__ constexpr int coupling_warps(int lam) { return lam <= 5 ? 1 : (lam <= 8 ? 2 : 4); }

constexpr int kHalf = 16;         // columns of the harmonic table
constexpr int kHS = kHalf + 1;   // its row stride: odd, so that 8-byte loads of different rows fall in different banks; the
                                 // last word holds the row's codes (g_row) of the two sets of scales

// Global to shared memory without a register: the tables of a block arrive behind the first nuclei's loads.
template <int N>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"(N));
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int LAM>
struct Shape {
  static constexpr int nS = n_harm(LAM), nB = n_beta(LAM), nR = n_r(LAM), NW = coupling_warps(LAM);
  static constexpr int nK = NW == 1 ? (LAM + 1) * (LAM + 2) / 2 : 0;  // steps kept in shared memory, per set
  static constexpr size_t smem = 32 * (size_t)nK + 8 * (size_t)(nS * kHS + (nB + 3) * kCS + nR + nS + 4 * nB + (LAM + 1)) +
                                 4 * (size_t)(2 * nB + 2 * (LAM + 1) + 8);
};

// Column split over NW warps: warp w takes |m| in [column_bound(w), column_bound(w + 1)), the columns' steps evened out.
__host__ __device__ constexpr int column_bound(int lam, int nw, int w) {
  if (w <= 0) return 0;
  if (w >= nw) return lam + 1;
  const int total = (lam + 1) * (lam + 2) / 2;
  int m = 0, acc = 0;
  while (m <= lam && nw * (acc + (lam - m + 1) / 2) < w * total) acc += lam - m++ + 1;
  return m;
}

// Columns m = am (neg: -am), am in [A0, A1), of V_lm into rows h of St at column c: the two signs on the two halves of a
// warp, so that 16 nuclei fill it.
template <int LAM>
__device__ __forceinline__ void harmonic_half(int A0, int A1, const int4* steps, bool neg, fx x, fx y, fx z, int2* St, int c) {
  fx dp = {1 << kFxLimb, 0}, dm = {0, 0};  // (x + iy)^am
  const fx ny = fx_neg(y);
#pragma unroll 1
  for (int am = 0; am < A1; ++am) {
    if (am >= A0) {
      fx v0 = {0, 0}, v1 = neg ? dm : dp;
      const int sm = neg ? -am : am;
#pragma unroll 1
      for (int l = am;; ++l) {
        if (!neg || am) St[(l * l + l + sm) * kHS + c] = make_int2(v1.h, v1.l);
        if (l == LAM) break;
        const int4 s = steps[l * (l + 1) / 2 + am];
        const fx vn = fx_step(fx{z.h << s.z, z.l << s.z}, v1, s.x, s.y, v0);
        v0 = v1;
        v1 = vn;
      }
    }
    const fx t = fx_step(x, dp, ny.h, ny.l, dm);
    dm = fx_step(y, dp, x.h, x.l, dm);
    dp = t;
  }
}

template <int LAM>
__global__ void __launch_bounds__(32 * coupling_warps(LAM)) k_coupling_fp64(CouplingArgs A) {
  using Sh = Shape<LAM>;
  constexpr int NW = Sh::NW, NT = 32 * NW, nS = Sh::nS, nB = Sh::nB, nR = Sh::nR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int4* Ks = reinterpret_cast<int4*>(smem_raw);             // [2][nK] steps of the harmonics
  int2* St = reinterpret_cast<int2*>(Ks + 2 * Sh::nK);             // [nS] harmonic rows of 16 columns
  int2* Bt = St + nS * kHS;                                  // [nB] radial rows (doubles, then fixed point but on the axis)
  int2* Xt = Bt + nB * kCS;                                  // [3] x, y, z of the columns
  double* nacc = reinterpret_cast<double*>(Xt + 3 * kCS);    // [nR] near sums
  double* fard = nacc + nR;                                  // [nS] far sums
  double* axs = fard + nS;                                   // [nB] axis sums
  double* sb = axs + nB;                                     // [nB] 2 pi k! p^{-(k+1)-L/2}
  double* cfa = sb + nB;                                     // [nB] a_{L,k}
  double* cfk = cfa + nB;                                    // [nB] 2 pi k!
  double* pw = cfk + nB;                                     // [LAM + 1] p^{-1-j/2}
  int* en = reinterpret_cast<int*>(pw + LAM + 1);            // [nB] biased exponent of the near columns of a row
  int* blk = en + nB;                                        // [nB] L | (L + 2k) << 8
  int* ef = blk + nB;                                        // [LAM + 1] the same of the far columns
  int* b0 = ef + LAM + 1;                                    // [LAM + 1] first radial row of L
  int* cnt = b0 + LAM + 1;                                   // near end, far end, near-axis end, columns, exponent of x, y
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  __shared__ long long s_next[2];
  __shared__ unsigned long long s_t0;
  constexpr int cb1 = column_bound(LAM, NW, 1), cb2 = column_bound(LAM, NW, 2), cb3 = column_bound(LAM, NW, 3);
  const int A0 = wid == 0 ? 0 : (wid == 1 ? cb1 : (wid == 2 ? cb2 : cb3));
  const int A1 = wid == NW - 1 ? LAM + 1 : (wid == 0 ? cb1 : (wid == 1 ? cb2 : cb3));
  // one radial row per thread, so that the loads of all rows are in flight together instead of one after another per L
  // (V of 32 atoms with l <= 6 378 -> 372 us, of 5 such atoms 100 -> 95 us, 9 atoms with l <= 3 46.5 -> 45.4 us)
  for (int b = tid; b < nB; b += NT) {
    int L = 0, k = b;
    for (int n = LAM / 2 + 1; k >= n; n = (LAM - L) / 2 + 1) {
      k -= n;
      ++L;
    }
    if (k == 0) b0[L] = b;
    blk[b] = L | (L + 2 * k) << 8;
    copy_async<8>(cfa + b, g_far + L * (kLamDer / 2 + 1) + k);
    copy_async<8>(cfk + b, g_kfact + k);
  }
  // the tables of a block: a small call is one block's chain of dependent instructions and cold loads per launch, so none of
  // these loads is waited for before the first nuclei's own
  for (int k = tid; k < 2 * Sh::nK; k += NT) copy_async<16>(Ks + k, g_step + (k < Sh::nK ? k : kSteps + k - Sh::nK));
  for (int h = tid; h < nS; h += NT) {
    int2* code = St + h * kHS + kHalf;
    copy_async<4>(&code->x, g_row + h);
    copy_async<4>(&code->y, g_row + kRows + h);
  }
  // a block takes A.group consecutive primitive pairs at a time, which mostly share their shell pair: the nuclei's
  // pair-frame coordinates (13 of some 80 FP64 instructions at small Lambda) are then formed once for the shell pair
  WorkQueue groups = A.q;
  groups.items = nullptr;
  wq_for_each(groups, (A.npp + A.group - 1) / A.group, s_next, &s_t0, [&](long long g) {
    double gx = 0.0, gy = 0.0, gz = 0.0, gq = 0.0;  // coordinates and charge of nucleus `lane` for shell pair gpr
    int gpr = -1;
    for (int64_t i = g * A.group; i < min(A.npp, (int64_t)(g + 1) * A.group); ++i) {
      const int64_t w = A.q.items ? A.q.items[i] : i;
      const int64_t q = A.pp_base + w;
      const int pr = A.pp_pair[q];
      const PPData pd = A.ppd[q];
      // primitive pairs with a zero prefactor (K_AB of Eq. 5 underflowed, or the pair is below the per-basis bound) are
      // skipped by the pair kernel too, so their coupling block is not needed
      if (pd.pref == 0.0) continue;
      const double ip = pd.sp * pd.rp;  // p^{-1/2}
      int64_t cbeg, ncen;
      mol_centers(A.mv, pr, cbeg, ncen);
      bool havenear = false, havefar = false;
      for (int64_t c0 = 0; c0 < ncen || c0 == 0; c0 += kNch) {
        __syncthreads();  // the tables of the previous chunk (or primitive pair) are consumed
        if (wid == NW - 1 && c0 == 0 && lane <= LAM) {  // p^{-1-j/2}, lane = j
          double v = pd.rp, b = ip;
#pragma unroll
          for (int bit = 0; (1 << bit) <= LAM; ++bit) {
            if ((lane >> bit) & 1) v *= b;
            b *= b;
          }
          pw[lane] = v;
        }
        if (wid == 0) {
          const bool valid = c0 + lane < ncen;
          if (pr != gpr || ncen > kNch) {
            gx = gy = gz = gq = 0.0;
            if (valid) {
              const int64_t c = mol_center_index(A.mv, cbeg + c0 + lane);
              // C - P = (C - A) - (beta/p)(B - A), in the pair frame where B - A is along z
              frame_coords(A.site_rot + 9 * (int64_t)A.pair_site[pr], A.shell_xyz + 3 * (int64_t)A.pair_a[pr],
                           A.centers + 3 * c, gx, gy, gz);
              gq = A.charges[c];
            }
            gpr = pr;
          }
          const double dx = gx, dy = gy, zp = gz;
          double Z = gq;
          const double dz = zp - pd.shift;
          const double rho2 = fma(dy, dy, dx * dx), s2 = fma(dz, dz, rho2), T = pd.p * s2;
          const int hs = __double2hiint(s2);
          if ((hs & 0x7ff00000) == 0x7ff00000) Z = __longlong_as_double(0x7ff8000000000000ll);  // no finite distance
          double ri = 0.0, ux = 0.0, uy = 0.0, uz = 1.0;
          if (hs >= kTinyHi) {
            ri = rsqrt(s2);
            ux = dx * ri;
            uy = dy * ri;
            uz = dz * ri;
          }
          // on the A-B line to within rounding of the rotation: rho below 2^-48 of |z_C - z_A|
          const int erho = (__double2hiint(rho2) >> 20) & 0x7ff, ezp = (__double2hiint(zp) >> 20) & 0x7ff;
          const bool axis = hs < 0x7ff00000 && (ri == 0.0 || erho == 0 || erho + 96 + 1023 < 2 * ezp);
          constexpr double kFar = far_t(LAM);
          const bool near = __double2hiint(T) < __double2hiint(kFar);
          const unsigned mn = __ballot_sync(~0u, valid && near && !axis), mf = __ballot_sync(~0u, valid && !near && !axis);
          const unsigned an = __ballot_sync(~0u, valid && near && axis), af = __ballot_sync(~0u, valid && !near && axis);
          const int n1 = __popc(mn), n2 = n1 + __popc(mf), n3 = n2 + __popc(an), n4 = n3 + __popc(af);
          const unsigned below = (1u << lane) - 1u;
          const int pos = axis ? (near ? n2 + __popc(an & below) : n3 + __popc(af & below))
                               : (near ? __popc(mn & below) : n1 + __popc(mf & below));
          // scale of x and y: the power of two of the largest in the chunk
          const bool off = valid && !axis;
          const unsigned hxy = max(__double2hiint(ux) & 0x7fffffff, __double2hiint(uy) & 0x7fffffff);
          const int exy = (int)(__reduce_max_sync(~0u, off ? hxy : 0u) >> 20) - 1023;
          const int er = exy >= -1 ? 0 : exy + 2;
          if (off) {
            const fx fxx = fx_of(ux, 1023 + er), fxy = fx_of(uy, 1023 + er), fxz = fx_of(uz, 1023);
            Xt[pos] = make_int2(fxx.h, fxx.l);
            Xt[kCS + pos] = make_int2(fxy.h, fxy.l);
            Xt[2 * kCS + pos] = make_int2(fxz.h, fxz.l);
          }
          if (lane == 0) {
            cnt[0] = n1;
            cnt[1] = n2;
            cnt[2] = n3;
            cnt[3] = n4;
            cnt[4] = er;
          }
          double G[LAM + 1], tau[LAM / 2 + 1];
          radial_factors<LAM>(near, T, pd.sp * (s2 * ri), ri * ip, Z,
                              g_boys_top + (size_t)LAM * kBoysTopRows * (kBoysTopStride / 2), G, tau);
          const bool anynear = (mn | an) != 0u;
          const int sgn = uz < 0.0 ? (int)0x80000000 : 0;
          int bo = 0;
#pragma unroll
          for (int L = 0; L <= LAM; ++L) {
            double acc = G[L];
#pragma unroll
            for (int k = 0; k <= (LAM - L) / 2; ++k) {
              if (k > 0 && !anynear) break;
              if (k > 0) acc = fma(tau[k], G[L + k], acc);
              const unsigned ha = (unsigned)__double2hiint(acc) & 0x7fffffffu;
              const int En = (int)(__reduce_max_sync(~0u, near && off ? ha : 0u) >> 20);
              if (k == 0) {
                const int Ef = (int)(__reduce_max_sync(~0u, !near && off ? ha : 0u) >> 20);
                if (lane == 0) ef[L] = Ef;
              }
              if (lane == 0) en[bo + k] = En;
              // U_L0(0, 0, +-1) N_L0 = (+-1)^L on the axis
              if (valid && (near || k == 0))
                Bt[(bo + k) * kCS + pos] =
                    make_int2(__double2loint(acc), __double2hiint(acc) ^ (axis && (L & 1) ? sgn : 0));
            }
            bo += (LAM - L) / 2 + 1;
          }
        }
        copy_wait();  // the block's tables, on its first primitive pair
        __syncthreads();
        const int n1 = cnt[0], n2 = cnt[1], n3 = cnt[2], n4 = cnt[3], er = cnt[4];
        const int4* steps = NW == 1 ? Ks + (er < 0 ? Sh::nK : 0) : k_step + (er < 0 ? kSteps : 0);
        const int col = lane & (kHalf - 1);
        const int* rowcode = reinterpret_cast<const int*>(St + kHalf) + (er < 0 ? 1 : 0);  // row h at 2 h kHS
        auto columns = [&](int h0) {
          const int c = h0 + col;
          if (c < n2) {
            const int2 a = Xt[c], b = Xt[kCS + c], z = Xt[2 * kCS + c];
            harmonic_half<LAM>(A0, A1, steps, lane >= kHalf, fx{a.x, a.y}, fx{b.x, b.y}, fx{z.x, z.y}, St, col);
          }
        };
        // radial rows into fixed point, lane = column
        for (int b = wid; b < nB; b += NW) {
          const int L = blk[b] & 0xff;
          const bool lead = b == b0[L];
          if (lane < n1 || (lead && lane < n2)) {
            int2* v = Bt + b * kCS + lane;
            // below 2^57: the sums of 16 products stay inside 64 bits
            const fx f = fx_of(__hiloint2double(v->y, v->x), (lane < n1 ? en[b] : ef[L]) + 2);
            *v = make_int2(f.h, f.l);
          }
        }
        columns(0);
        // axis sums of the radial rows and the rows' scales
        for (int b = tid; b < nB; b += NT) {
          double s = c0 == 0 ? 0.0 : axs[b];
          for (int c = n2; c < n3; ++c) {
            const int2 v = Bt[b * kCS + c];
            s += __hiloint2double(v.y, v.x);
          }
          if (n3 < n4) {
            const int2* row = Bt + b0[blk[b] & 0xff] * kCS;
            double f = 0.0;
            for (int c = n3; c < n4; ++c) f += __hiloint2double(row[c].y, row[c].x);
            s = fma(f, cfa[b], s);
          }
          axs[b] = s;
          if (c0 == 0) sb[b] = cfk[b] * pw[blk[b] >> 8];
        }
        __syncthreads();
        for (int h0 = 0; h0 < n2; h0 += kHalf) {
          if (h0 > 0) {
            __syncthreads();  // the first half's harmonics are consumed
            columns(h0);
            __syncthreads();
          }
          const int hn = min(n1, h0 + kHalf), hf = min(n2, h0 + kHalf), f0 = max(n1, h0);
          if (f0 < hf) {
            for (int h = tid; h < nS; h += NT) {
              const int code = rowcode[2 * h * kHS], L = code >> 16;
              const int2 *s = St + h * kHS - h0, *b = Bt + b0[L] * kCS;
              long long hh = 0, mid = 0;
#pragma unroll (NW == 1 ? 1 : 4)  // short code where a warp is alone: each launch fetches it anew
              for (int c = f0; c < hf; ++c) {
                const int2 u = s[c], v = b[c];
                hh = fx_mad(u.x, v.x, hh);
                mid = fx_mad(u.x, v.y, mid);
                mid = fx_mad(u.y, v.x, mid);
              }
              const int E = ef[L];
              const double v = E == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                          : fx_double(fx_sum(hh, mid),
                                                      E + 2 - 1023 - kFxBits + er * (code & 0xff) - ((code >> 8) & 0xff));
              fard[h] = havefar ? fard[h] + v : v;
            }
            havefar = true;
          }
          if (h0 < hn) {
            for (int e = tid; e < nR; e += NT) {
              const int code = __ldg(A.rmap + e), h = code & 0xfff, b = (code >> 12) & 0xfff;
              const int rc = rowcode[2 * h * kHS];
              const int2 *s = St + h * kHS - h0, *r = Bt + b * kCS;
              long long hh = 0, mid = 0;
#pragma unroll (NW == 1 ? 1 : 4)  // short code where a warp is alone: each launch fetches it anew
              for (int c = h0; c < hn; ++c) {
                const int2 u = s[c], x = r[c];
                hh = fx_mad(u.x, x.x, hh);
                mid = fx_mad(u.x, x.y, mid);
                mid = fx_mad(u.y, x.x, mid);
              }
              const int E = en[b];
              const double v = E == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                          : fx_double(fx_sum(hh, mid),
                                                      E + 2 - 1023 - kFxBits + er * (rc & 0xff) - ((rc >> 8) & 0xff));
              nacc[e] = havenear ? nacc[e] + v : v;
            }
            havenear = true;
          }
        }
      }
      __syncthreads();
      double* out = A.rbuf + A.rbase + w * (int64_t)nR;
      for (int e = tid; e < nR; e += NT) {
        const int code = __ldg(A.rmap + e), h = code & 0xfff, b = (code >> 12) & 0xfff;
        double v = havenear ? nacc[e] : 0.0;
        if (havefar) v = fma(fard[h], cfa[b], v);
        out[e] = fma(v, __ldg(A.rnorm + e), (St[h * kHS + kHalf].x & 0xff) == 0 ? axs[b] : 0.0) * sb[b];
      }
    }
  });
  copy_wait();
}

using CouplingKernel = void (*)(CouplingArgs);

template <int... L>
constexpr CouplingKernel kernel_at(int lam, std::integer_sequence<int, L...>) {
  CouplingKernel k = nullptr;
  ((lam == L ? (k = &k_coupling_fp64<L>, 0) : 0), ...);
  return k;
}

template <int... L>
constexpr size_t smem_at(int lam, std::integer_sequence<int, L...>) {
  size_t s = 0;
  ((lam == L ? (s = Shape<L>::smem, 0) : 0), ...);
  return s;
}

using Lams = std::make_integer_sequence<int, kLamDer + 1>;  // derivative integrals run at la + lb + 1

}  // namespace

cudaError_t coupling_fp64_setup() {
  cudaError_t e = upload_nucleus_constants();
  const std::vector<double>& bt = tables_host().boys_top;
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_boys_top, bt.data(), sizeof(double) * bt.size());
  for (int lam = 0; lam <= kLamDer && e == cudaSuccess; ++lam)
    e = set_max_dynamic_smem((const void*)kernel_at(lam, Lams{}));
  return e;
}

cudaError_t boys_top_table(int lam, const double2** out) {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_boys_top);
  *out = static_cast<const double2*>(p) + (size_t)lam * kBoysTopRows * (kBoysTopStride / 2);
  return e;
}

cudaError_t launch_coupling_fp64(int lam, const CouplingArgs& args, cudaStream_t stream) {
  if (lam < 0 || lam > kLamDer) return cudaErrorInvalidValue;
  // up to 32 one-warp blocks per SM (the block limit), half of it where a block has two or four warps; primitive pairs
  // are taken four at a time once that leaves every SM eight rounds or more (no result depends on it)
  const int nw = coupling_warps(lam), per_sm = nw == 1 ? 32 : 16;
  CouplingArgs a = args;
  a.group = args.npp >= (int64_t)152 * per_sm * 8 ? 4 : 1;
  kernel_at(lam, Lams{})<<<grid_cap_sm((args.npp + a.group - 1) / a.group, per_sm), 32 * nw, smem_at(lam, Lams{}), stream>>>(a);
  return cudaGetLastError();
}

}  // namespace shgo
