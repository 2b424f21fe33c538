// Electrostatic potential of a density at arbitrary points and its gradient (FP64): phi(x) = sum_ab D_ab <a|1/|r-x||b>.
//
// The pair kernel is a linear map from the nucleus sums of each primitive pair to V; its adjoint, once per density
// (k_esp_adjoint), maps each density block back to weights W of every primitive pair, so that with the tables of the
// coupling kernel (shgo_nucleus.cuh; d = x - P in the pair frame, u = d/|d|, t = sqrt(p) |d|)
//   phi(x) = sum_pp sum_{L,M,k} W[L,M,k] U_LM(u) b_{L,k}(t).
// The gradient is the same form: d/dx of the integral of f(r - P)/|r - x| is that of the gradient of f, whose
// one-centre parts are fixed combinations of order Lambda + 1 (Tables::d_field, d_raise), so the adjoint of that step and
// the rotation to the molecular frame give three sets of weights of order Lambda + 1, summed against one set of tables.
// Far away that sum over the rows of a degree cancels down to the degrees L + 1 (t^2 in accuracy: 5e-12 of a p-s pair's
// gradient at p = 100, 20 bohr off), so the far weights of the gradient come from those of the potential instead, by the
// derivative of S_LM(d) / |d|^{2L+1} (Tables::fr_terms; 3e-16 there, 1 % of the call of 251 points).
//
// What bounds it: as in the coupling kernel FP64 (1.7 lanes per clock and SM) is kept for the geometry, the radial
// values and one multiply-add per radial row; the harmonics and the sums over M run in 58-bit fixed point on the integer
// pipe.  Points far from P (T >= far_t: nearly all of a grid at ordinary exponents) have b_{L,k} = a_{L,k} t^{-(L+1)}:
// weights summed over k beforehand, Lambda + 1 rows instead of one per (L, k), no Boys values.  A block takes 128 points,
// so that near and far points of one primitive pair fill separate groups of 32 lanes; the classes run concurrently.
//
// Measured (GB300, basis of 32 atoms with l <= 6, against FP64 tables per 32 points and per-entry sums, four harmonic
// tables for the gradient): 2003 points 27.9 -> 6.6 ms, gradient at 251 points 19.7 -> 2.3 ms (1.1 of them the adjoint),
// the errors against 64-bit quadrature unchanged.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <string>
#include <utility>
#include <vector>

#include "shgo_internal.h"
#include "shgo_nucleus.cuh"

namespace shgo {

namespace {

constexpr int kPts = 128;    // points per block, one per thread in the geometry phase
constexpr int kEspWarps = 4;

// Weights of one primitive pair, in 8-byte words: per component the limbs of W[e] (near) and of sum_k a_{L,k} W[L,M,k]
// (far), then the biased exponents of the near rows (L, k) and of the far rows L.
__host__ __device__ constexpr int weight_words(int lam, int nc) {
  return nc * (n_r(lam) + n_harm(lam)) + (nc * (n_beta(lam) + lam + 1) + 1) / 2;
}

struct EspArgs {
  int64_t npp = 0, pp_base = 0;  // primitive pairs of the piece
  const int* pp_pair = nullptr;
  const int* pair_a = nullptr;
  const double* shell_xyz = nullptr;
  const double* site_rot = nullptr;
  const int* pair_site = nullptr;
  const PPData* ppd = nullptr;
  const double2* boys_top = nullptr;
  const int2* weights = nullptr;
  int64_t npoints = 0;
  const double* points = nullptr;
  double* phi = nullptr;
  int nchunks = 0, nsplit = 0;  // blocks = nchunks x nsplit
};

template <int LAM, int NC>
struct EspShape {
  static constexpr int nS = n_harm(LAM), nB = n_beta(LAM), nR = n_r(LAM);
  static constexpr size_t smem =
      8 * (size_t)((nS + nB) * kCS + NC * (nR + nS) + 5 * kPts + NC * kPts + kEspWarps * NC * 32) +
      4 * (size_t)(NC * (nB + LAM + 1) + nB + 2 * (LAM + 1) + kPts + 2 * kEspWarps);
};

// Column split of the harmonics over the warps w0 .. 3 (warp 0 evaluates the near points' radial rows meanwhile).
__host__ __device__ constexpr int esp_column_bound(int lam, int nw, int w) {
  if (w <= 0) return 0;
  if (w >= nw) return lam + 1;
  const int total = (lam + 1) * (lam + 1);
  int m = 0, acc = 0;
  while (m <= lam && nw * (acc + (lam - m + 1) * (m ? 2 : 1) / 2) < w * total) {
    acc += (lam - m + 1) * (m ? 2 : 1);
    ++m;
  }
  return m;
}

// One block: a chunk of 128 points and every nsplit-th primitive pair.  Per primitive pair each thread places its point
// in the near or the far list; groups of 32 of one list then run: radial rows (warp 0) beside the harmonic columns,
// then the rows' sums over M, rows dealt to the warps, lane = point.
template <int LAM, int NC>
__global__ void __launch_bounds__(32 * kEspWarps) k_esp(EspArgs A) {
  using Sh = EspShape<LAM, NC>;
  constexpr int nS = Sh::nS, nB = Sh::nB, nR = Sh::nR, WW = weight_words(LAM, NC);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int2* St = reinterpret_cast<int2*>(smem_raw);            // [nS] harmonic rows of the group
  double* Bd = reinterpret_cast<double*>(St + nS * kCS);    // [nB] radial rows of the group
  int2* wn = reinterpret_cast<int2*>(Bd + nB * kCS);        // [NC][nR] near weights
  int2* wf = wn + NC * nR;                                  // [NC][nS] far weights
  int2* Xs = wf + NC * nS;                                  // [3][kPts] u of the listed points
  double* tt = reinterpret_cast<double*>(Xs + 3 * kPts);    // [kPts] near: t, far: 1/t
  double* TT = tt + kPts;                                   // [kPts] T
  double* acc = TT + kPts;                                  // [NC][kPts] sums of the block's points
  double* part = acc + NC * kPts;                           // [warps][NC][32]
  int* ew = reinterpret_cast<int*>(part + kEspWarps * NC * 32);  // [NC][nB], [NC][LAM + 1] exponents
  int* rows = ew + NC * (nB + LAM + 1);                     // [nB] L | k << 8
  int* b0 = rows + nB;                                      // [LAM + 1] first radial row of L
  int* rb = b0 + LAM + 1;                                   // [LAM + 1] first entry of L
  int* idx = rb + LAM + 1;                                  // [kPts] point of a list slot
  int* cnts = idx + kPts;                                   // near and far counts of the warps
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int chunk = blockIdx.x % A.nchunks, split = blockIdx.x / A.nchunks;
  const int64_t pt = (int64_t)chunk * kPts + tid;
  const bool valid = pt < A.npoints;
  for (int L = tid; L <= LAM; L += 32 * kEspWarps) {
    const int f = beta_first(LAM, L), nk = (LAM - L) / 2 + 1;
    int r = 0;
    for (int l = 0; l < L; ++l) r += (2 * l + 1) * ((LAM - l) / 2 + 1);
    b0[L] = f;
    rb[L] = r;
    for (int k = 0; k < nk; ++k) rows[f + k] = L | k << 8;
  }
  double xp[3] = {0.0, 0.0, 0.0};
  if (valid)
    for (int k = 0; k < 3; ++k) xp[k] = A.points[3 * pt + k];
  for (int c = 0; c < NC; ++c) acc[c * kPts + tid] = 0.0;
  constexpr int f1 = esp_column_bound(LAM, 4, 1), f2 = esp_column_bound(LAM, 4, 2), f3 = esp_column_bound(LAM, 4, 3);
  constexpr int g1 = esp_column_bound(LAM, 3, 1), g2 = esp_column_bound(LAM, 3, 2);
  const int fa0 = wid == 0 ? 0 : (wid == 1 ? f1 : (wid == 2 ? f2 : f3));
  const int fa1 = wid == 0 ? f1 : (wid == 1 ? f2 : (wid == 2 ? f3 : LAM + 1));
  const int na0 = wid <= 1 ? 0 : (wid == 2 ? g1 : g2), na1 = wid == 0 ? 0 : (wid == 1 ? g1 : (wid == 2 ? g2 : LAM + 1));
  for (int64_t w = split; w < A.npp; w += A.nsplit) {
    const int64_t q = A.pp_base + w;
    const PPData pd = A.ppd[q];
    if (pd.pref == 0.0) continue;  // uniform over the block
    const int pr = A.pp_pair[q];
    __syncthreads();  // the previous primitive pair's weights and lists are consumed
    const int2* src = A.weights + w * WW;
    for (int e = tid; e < NC * (nR + nS); e += 32 * kEspWarps) wn[e] = __ldg(src + e);
    const int* esrc = reinterpret_cast<const int*>(src + NC * (nR + nS));
    for (int e = tid; e < NC * (nB + LAM + 1); e += 32 * kEspWarps) ew[e] = __ldg(esrc + e);
    double x, y, z;
    frame_coords(A.site_rot + 9 * (int64_t)A.pair_site[pr], A.shell_xyz + 3 * (int64_t)A.pair_a[pr], xp, x, y, z);
    z -= pd.shift;
    const double s2 = fma(z, z, fma(y, y, x * x)), T = pd.p * s2;
    double ri = 0.0, ux = 0.0, uy = 0.0, uz = 1.0;
    if (__double2hiint(s2) >= kTinyHi) {
      ri = rsqrt(s2);
      ux = x * ri;
      uy = y * ri;
      uz = z * ri;
    }
    constexpr double kFar = far_t(LAM);
    const bool near = __double2hiint(T) < __double2hiint(kFar);
    const unsigned mn = __ballot_sync(~0u, valid && near), mf = __ballot_sync(~0u, valid && !near);
    if (lane == 0) {
      cnts[wid] = __popc(mn);
      cnts[kEspWarps + wid] = __popc(mf);
    }
    __syncthreads();
    int NN = 0, NF = 0, bn = 0, bf = 0;
#pragma unroll
    for (int k = 0; k < kEspWarps; ++k) {
      if (k < wid) {
        bn += cnts[k];
        bf += cnts[kEspWarps + k];
      }
      NN += cnts[k];
      NF += cnts[kEspWarps + k];
    }
    if (valid) {
      const unsigned below = (1u << lane) - 1u;
      const int slot = near ? bn + __popc(mn & below) : NN + bf + __popc(mf & below);
      const fx a = fx_of(ux, 1023), b = fx_of(uy, 1023), c = fx_of(uz, 1023);
      Xs[slot] = make_int2(a.h, a.l);
      Xs[kPts + slot] = make_int2(b.h, b.l);
      Xs[2 * kPts + slot] = make_int2(c.h, c.l);
      tt[slot] = near ? pd.sp * (s2 * ri) : ri * (pd.sp * pd.rp);
      TT[slot] = T;
      idx[slot] = tid;
    }
    __syncthreads();
    for (int s0 = 0; s0 < NN + NF;) {
      const bool ng = s0 < NN;
      const int cnt = min(32, (ng ? NN : NN + NF) - s0);
      if (wid == 0 && lane < cnt) {
        double G[LAM + 1], tau[LAM / 2 + 1];
        const double t = tt[s0 + lane];
        radial_factors<LAM>(ng, TT[s0 + lane], t, t, 1.0, A.boys_top, G, tau);
        if (ng) {
          int bo = 0;
#pragma unroll
          for (int L = 0; L <= LAM; ++L) {
            double s = G[L];
            Bd[bo * kCS + lane] = s;
#pragma unroll
            for (int k = 1; k <= (LAM - L) / 2; ++k) {
              s = fma(tau[k], G[L + k], s);
              Bd[(bo + k) * kCS + lane] = s;
            }
            bo += (LAM - L) / 2 + 1;
          }
        } else {
#pragma unroll
          for (int L = 0; L <= LAM; ++L) Bd[L * kCS + lane] = G[L];
        }
      }
      if (lane < cnt) {
        const int2 a = Xs[s0 + lane], b = Xs[kPts + s0 + lane], c = Xs[2 * kPts + s0 + lane];
        harmonic_columns<LAM>(ng ? na0 : fa0, ng ? na1 : fa1, 0, fx{a.x, a.y}, fx{b.x, b.y}, fx{c.x, c.y}, St, lane);
      }
      __syncthreads();
      double r[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) r[c] = 0.0;
      const int nrow = ng ? nB : LAM + 1;
      for (int j = wid; j < nrow; j += kEspWarps) {
        const int L = ng ? rows[j] & 0xff : j, nk = ng ? (LAM - L) / 2 + 1 : 1;
        const int2* wp = ng ? wn + rb[L] + (rows[j] >> 8) : wf + L * L;
        const int2* sp = St + L * L * kCS + lane;
        const int ws = ng ? nR : nS;
        long long hh[NC], mid[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) hh[c] = mid[c] = 0;
#pragma unroll 4
        for (int m = 0; m <= 2 * L; ++m) {
          const int2 v = sp[m * kCS];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const int2 g = wp[c * ws + m * nk];
            hh[c] = fx_mad(v.x, g.x, hh[c]);
            mid[c] = fx_mad(v.x, g.y, mid[c]);
            mid[c] = fx_mad(v.y, g.x, mid[c]);
          }
        }
        const double b = Bd[j * kCS + lane];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int E = ng ? ew[c * nB + j] : ew[NC * nB + c * (LAM + 1) + j];
          const double s = E == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                      : fx_double(fx_sum(hh[c], mid[c]), E + 2 - 1023 - kFxBits);
          r[c] = fma(s, b, r[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) part[(wid * NC + c) * 32 + lane] = r[c];
      __syncthreads();
      if (wid == 0 && lane < cnt) {
        const int i = idx[s0 + lane];
#pragma unroll
        for (int c = 0; c < NC; ++c)
          acc[c * kPts + i] += (part[c * 32 + lane] + part[(NC + c) * 32 + lane]) +
                               (part[(2 * NC + c) * 32 + lane] + part[(3 * NC + c) * 32 + lane]);
      }
      s0 += cnt;
    }
  }
  __syncthreads();
  if (valid)
    for (int c = 0; c < NC; ++c) atomicAdd(A.phi + NC * pt + c, acc[c * kPts + tid]);
}

// Adjoint of the pair kernel: for one shell pair and a symmetric density D, the weights of every primitive pair.  Steps
// reversed: the density block is rotated into the pair frame (D' = D^la^T D_blk D^lb), weighted by the translation
// factors (Wbar[l1 m1][l2 m2] = t_A(l1, m1) t_B(l2, m2) D'[m1][m2]), pulled back through the Gaunt coupling (transposed
// program, primitive factors), for the gradient through the transposed field step of each axis and the rotation of the
// axes, scaled by 2 pi k! p^{-(k+1)-L/2} N_LM, and written as fixed point with one exponent per row.
template <int NC>
__host__ __device__ inline size_t adjoint_smem(int la, int lb) {
  const int nWa = (la + 1) * (la + 1), na = 2 * la + 1, nb = 2 * lb + 1, lm = la > lb ? la : lb;
  const int lam1 = la + lb + (NC == 3 ? 1 : 0);
  return sizeof(double) * ((size_t)nWa * w_stride(lb) + na * na + nb * nb + (la + 1) * na + (lb + 1) * nb +
                           3 * na * nb + (la + 1) * (lb + 1) + lam1 + 1 + lm + 1 + 8 + n_r(la + lb) + (NC == 3 ? n_harm(la + lb) : 0) +
                           NC * (n_r(lam1) + n_harm(lam1))) +
         sizeof(int) * (size_t)(NC * (n_beta(lam1) + lam1 + 1) + 3 * (lam1 + 2) + 8);
}

struct AdjointArgs {
  int la, lb, npairs, pair_base;
  int64_t pp_base;
  const int *pair_a, *pair_b;
  const int64_t* pair_ppoff;
  const int* pair_site;
  int64_t rot_per;
  const double *rotd, *site_rot;
  const int* shell_nprim;
  const int64_t* shell_foff;
  const double* etab;
  const int* eoff;
  const int* gt_ptr;
  const GTerm* gt_terms;
  const int* dt_ptr;       // transposed field step of la + lb (gradient)
  const GTerm* dt_terms;
  const GTerm* fr_terms;   // derivative of the far field (gradient)
  const int* rmap;         // layout of the weights' order
  const double* rnorm;
  const PPData* ppd;
  const double* D;
  int64_t ld;
  int2* weights;
};

template <int NC>
__global__ void __launch_bounds__(128) k_esp_adjoint(AdjointArgs A) {
  extern __shared__ double smem[];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int la = A.la, lb = A.lb, lam = la + lb, nR0 = n_r(lam);
  const int lam1 = lam + (NC == 3 ? 1 : 0), nR = n_r(lam1), nS = n_harm(lam1), nB = n_beta(lam1);
  const int nWa = (la + 1) * (la + 1), ws = w_stride(lb), nWs = nWa * ws;
  const int na = 2 * la + 1, nb = 2 * lb + 1;
  const int lm = la > lb ? la : lb;
  const int nDb = la != lb ? nb * nb : 0;
  double* Wb = smem;                       // [l1 m1][l2 m2], row stride ws
  double* Dm = Wb + nWs;                   // D^la, then D^lb when lb != la
  double* tA = Dm + na * na + nb * nb;
  double* tB = tA + (la + 1) * na;
  double* Db = tB + (lb + 1) * nb;         // density block [ma][mb]
  double* Y = Db + na * nb;
  double* Dp = Y + na * nb;                // pair-frame density
  double* fab = Dp + na * nb;
  double* pw = fab + (la + 1) * (lb + 1);  // p^{-1-j/2}
  double* dpow = pw + lam1 + 1;
  double* scal = dpow + lm + 1;
  double* g0 = scal + 8;                   // [nR0] weights of the unscaled coupling block
  double* qf = g0 + nR0;                   // [n_harm(lam)] far field of the coupling block (gradient)
  double* fin = qf + (NC == 3 ? n_harm(lam) : 0);  // [NC][nR] weights
  double* far = fin + NC * nR;             // [NC][nS] weights of the far points
  int* ex = reinterpret_cast<int*>(far + NC * nS);  // [NC][nB], [NC][lam1 + 1] biased exponents
  int* b0 = ex + NC * (nB + lam1 + 1);     // first radial row of L
  int* rb = b0 + lam1 + 2;                 // first entry of L
  const int* rowcode = g_row;
  if (tid == 0) {
    int b = 0, r = 0;
    for (int L = 0; L <= lam1 + 1; ++L) {
      b0[L] = b;
      rb[L] = r;
      if (L <= lam1) {
        b += (lam1 - L) / 2 + 1;
        r += (2 * L + 1) * ((lam1 - L) / 2 + 1);
      }
    }
  }
  for (int w = blockIdx.x; w < A.npairs; w += gridDim.x) {
    const int pr = A.pair_base + w;
    const int a = A.pair_a[pr], b = A.pair_b[pr];
    const double* rd = A.rotd + (int64_t)A.pair_site[pr] * A.rot_per;
    const double* Q = A.site_rot + 9 * (int64_t)A.pair_site[pr];
    const int64_t fa0 = A.shell_foff[a], fb0 = A.shell_foff[b];
    __syncthreads();
    if (tid == 0) {
      double v = 1.0;
      for (int k = 0; k <= lm; ++k) {
        dpow[k] = v;
        v *= rd[0];
      }
    }
    for (int e = tid; e < na * na; e += nth) Dm[e] = rd[1 + rot_doff(la) + e];
    for (int e = tid; e < nDb; e += nth) Dm[na * na + e] = rd[1 + rot_doff(lb) + e];
    for (int e = tid; e < na * nb; e += nth) {
      const int ma = e / nb, mb = e % nb;
      double v = A.D[(fa0 + ma) * A.ld + fb0 + mb];
      if (a != b) v += A.D[(fb0 + mb) * A.ld + fa0 + ma];
      Db[e] = v;
    }
    __syncthreads();
    for (int e = tid; e < (la + 1) * na; e += nth) {
      const int l1 = e / na, ma = e % na - la, lr = la - l1;
      tA[e] = l1 >= (ma < 0 ? -ma : ma) ? A.etab[A.eoff[la] + translation_offset_dev(la, ma, l1, ma) + lr] * dpow[lr] : 0.0;
    }
    for (int e = tid; e < (lb + 1) * nb; e += nth) {
      const int l2 = e / nb, mb = e % nb - lb, lr = lb - l2;
      tB[e] = l2 >= (mb < 0 ? -mb : mb)
                  ? A.etab[A.eoff[lb] + translation_offset_dev(lb, mb, l2, mb) + lr] * ((lr & 1) ? -dpow[lr] : dpow[lr])
                  : 0.0;
    }
    const double* Da = Dm;
    const double* Dbr = la != lb ? Dm + na * na : Dm;
    // Y = D_blk D^lb, then D' = D^la^T Y
    for (int e = tid; e < na * nb; e += nth) {
      const int ma = e / nb, k = e % nb;
      double sacc = 0.0;
      for (int mb = 0; mb < nb; ++mb) sacc = fma(Db[ma * nb + mb], Dbr[mb * nb + k], sacc);
      Y[e] = sacc;
    }
    __syncthreads();
    for (int e = tid; e < na * nb; e += nth) {
      const int k = e / nb, k2 = e % nb;
      double sacc = 0.0;
      for (int ma = 0; ma < na; ++ma) sacc = fma(Da[ma * na + k], Y[ma * nb + k2], sacc);
      Dp[e] = sacc;
    }
    __syncthreads();
    for (int e = tid; e < nWs; e += nth) {
      const int i1 = e / ws, i2 = e % ws;
      double v = 0.0;
      if (i2 < (lb + 1) * (lb + 1)) {
        int l1 = 0, l2 = 0;
        while ((l1 + 1) * (l1 + 1) <= i1) ++l1;
        while ((l2 + 1) * (l2 + 1) <= i2) ++l2;
        const int m1 = i1 - l1 * l1 - l1, m2 = i2 - l2 * l2 - l2;
        v = tA[l1 * na + m1 + la] * tB[l2 * nb + m2 + lb] * Dp[(m1 + la) * nb + m2 + lb];
      }
      Wb[e] = v;
    }
    const int npp = A.shell_nprim[a] * A.shell_nprim[b];
    const int64_t q0 = A.pair_ppoff[pr];
    for (int ij = 0; ij < npp; ++ij) {
      const PPData pd = A.ppd[q0 + ij];
      if (pd.pref == 0.0) continue;  // uniform; skipped by the potential kernel as well
      __syncthreads();  // the previous primitive pair is done with the tables
      if (tid < (la + 1) * (lb + 1)) {
        const int l1 = tid / (lb + 1), l2 = tid % (lb + 1);
        double v = pd.pref;
        for (int k = 0; k < la - l1; ++k) v *= pd.ra;
        for (int k = 0; k < lb - l2; ++k) v *= pd.rb;
        fab[tid] = v;
      }
      if (tid <= lam1) {
        const double ip = pd.sp * pd.rp;
        double v = pd.rp;
        for (int k = 0; k < tid; ++k) v *= ip;
        pw[tid] = v;
      }
      __syncthreads();
      for (int e = tid; e < nR0; e += nth) {
        double acc = 0.0;
        for (int t = A.gt_ptr[e]; t < A.gt_ptr[e + 1]; ++t) {
          const GTerm gt = A.gt_terms[t];
          acc = fma(gt.coef * fab[gt.pad], Wb[gt.ridx], acc);
        }
        g0[e] = acc;
      }
      __syncthreads();
      for (int e = tid; e < nR; e += nth) {
        const int code = __ldg(A.rmap + e), k = (code >> 24) & 0xff, L = __ldg(rowcode + (code & 0xfff)) >> 16;
        const double sc = __ldg(A.rnorm + e) * (g_kfact[k] * pw[L + 2 * k]);
        if constexpr (NC == 1) {
          fin[e] = g0[e] * sc;
        } else {
          double h[3];
          for (int c = 0; c < 3; ++c) {
            double s = 0.0, r = 0.0;
            for (int t = A.dt_ptr[3 * e + c]; t < A.dt_ptr[3 * e + c + 1]; ++t) {
              const GTerm g = A.dt_terms[t];
              if (g.pad)
                r = fma(g.coef, g0[g.ridx], r);
              else
                s = fma(g.coef, g0[g.ridx], s);
            }
            h[c] = fma(-2.0 * pd.p, r, s) * sc;
          }
          // to the molecular frame: grad_x = Q^T grad_d
          for (int x = 0; x < 3; ++x) fin[x * nR + e] = Q[x] * h[0] + Q[3 + x] * h[1] + Q[6 + x] * h[2];
        }
      }
      if constexpr (NC == 3) {
        int r = 0, L = 0;  // first entry of degree L in g0
        for (int h = tid; h < n_harm(lam); h += nth) {
          for (; (L + 1) * (L + 1) <= h; ++L) r += (2 * L + 1) * ((lam - L) / 2 + 1);
          const int nk = (lam - L) / 2 + 1;
          const double* v = g0 + r + (h - L * L) * nk;
          double s = 0.0;
          for (int k = 0; k < nk; ++k) s = fma(g_far[L * (kLamDer / 2 + 1) + k] * (g_kfact[k] * pw[L + 2 * k]), v[k], s);
          qf[h] = s;
        }
      }
      __syncthreads();
      if constexpr (NC == 1) {
        for (int h = tid; h < nS; h += nth) {
          const int L = __ldg(rowcode + h) >> 16, nk = (lam1 - L) / 2 + 1;
          const double* v = fin + rb[L] + (h - L * L) * nk;
          double s = 0.0;
          for (int k = 0; k < nk; ++k) s = fma(g_far[L * (kLamDer / 2 + 1) + k], v[k], s);
          far[h] = s;
        }
      } else {
        // gradient of the far field sum q_LM S_LM(u) t^{-(L+1)}, which has degrees L + 1 alone (the sums over k of the
        // weights above hold degrees L - 1 as well, that cancel in exact arithmetic only: t^2 in accuracy)
        for (int h = tid; h < nS; h += nth) {
          const int L = __ldg(rowcode + h) >> 16;
          const double s = pd.sp * __ldg(A.rnorm + rb[L] + (h - L * L) * ((lam1 - L) / 2 + 1));
          double f[kFarSlots];
#pragma unroll
          for (int j = 0; j < kFarSlots; ++j) {
            const GTerm t = A.fr_terms[kFarSlots * h + j];
            f[j] = t.coef * qf[t.ridx];
          }
          const double gx = (f[0] + f[1]) * s, gy = (f[2] + f[3]) * s, gz = f[4] * s;
          for (int x = 0; x < 3; ++x) far[x * nS + h] = Q[x] * gx + Q[3 + x] * gy + Q[6 + x] * gz;
        }
      }
      __syncthreads();
      // exponent of each row: the largest of |W_M| 2^-e(L,M)
      for (int x = tid; x < NC * (nB + lam1 + 1); x += nth) {
        const bool nr = x < NC * nB;
        const int y = nr ? x : x - NC * nB, per = nr ? nB : lam1 + 1, c = y / per, j = y - c * per;
        int L = j, k = 0;
        if (nr) {
          L = 0;
          while (b0[L + 1] <= j) ++L;
          k = j - b0[L];
        }
        const int nk = nr ? (lam1 - L) / 2 + 1 : 1;
        const double* v = nr ? fin + c * nR + rb[L] + k : far + c * nS + L * L;
        int E = 0;
        for (int m = 0; m <= 2 * L; ++m) {
          const int e = (__double2hiint(v[m * nk]) >> 20) & 0x7ff;
          E = max(E, e == 0x7ff ? e : e - ((__ldg(rowcode + L * L + m) >> 8) & 0xff));
        }
        ex[x] = E;
      }
      __syncthreads();
      int2* out = A.weights + (q0 + ij - A.pp_base) * (int64_t)weight_words(lam1, NC);
      for (int x = tid; x < NC * nR; x += nth) {
        const int c = x / nR, e = x - c * nR, code = __ldg(A.rmap + e), rc = __ldg(rowcode + (code & 0xfff));
        const int E = ex[c * nB + ((code >> 12) & 0xfff)];
        const fx f = E > 0 ? fx_of(fin[x], E + 2 + ((rc >> 8) & 0xff)) : fx{0, 0};
        out[x] = make_int2(f.h, f.l);
      }
      for (int x = tid; x < NC * nS; x += nth) {
        const int c = x / nS, rc = __ldg(rowcode + x - c * nS), E = ex[NC * nB + c * (lam1 + 1) + (rc >> 16)];
        const fx f = E > 0 ? fx_of(far[x], E + 2 + ((rc >> 8) & 0xff)) : fx{0, 0};
        out[NC * nR + x] = make_int2(f.h, f.l);
      }
      int* eo = reinterpret_cast<int*>(out + NC * (nR + nS));
      for (int x = tid; x < NC * (nB + lam1 + 1); x += nth) eo[x] = ex[x];
    }
  }
}

using EspKernel = void (*)(EspArgs);

template <int NC, int... L>
constexpr EspKernel esp_kernel_at(int lam, std::integer_sequence<int, L...>) {
  EspKernel k = nullptr;
  ((lam == L + (NC == 3) ? (k = &k_esp<L + (NC == 3), NC>, 0) : 0), ...);
  return k;
}

template <int NC, int... L>
constexpr size_t esp_smem_at(int lam, std::integer_sequence<int, L...>) {
  size_t s = 0;
  ((lam == L + (NC == 3) ? (s = EspShape<L + (NC == 3), NC>::smem, 0) : 0), ...);
  return s;
}

using Lams = std::make_integer_sequence<int, kLamMax + 1>;

// Pieces of a class whose weights fit `words` 8-byte words, cut between shell pairs.
std::vector<ClassWork> pieces(const ClassWork& w, const int64_t* ppoff, int64_t per, int64_t words) {
  std::vector<ClassWork> out;
  const int qend = w.pair_base + w.npairs;
  for (int q = w.pair_base; q < qend;) {
    ClassWork c{w.la, w.lb, 0, q, 0, ppoff[q]};
    while (q < qend && (c.npairs == 0 || (ppoff[q + 1] - c.pp_base) * per <= words)) {
      ++c.npairs;
      ++q;
    }
    c.npp = ppoff[q] - c.pp_base;
    out.push_back(c);
  }
  return out;
}

// Weights of one piece, in 8-byte words, one region per pool stream: 64 MiB, so that the regions of all 16 streams stay
// within what the workspace pool keeps between calls (600 points of 150 atoms with l <= 6 take 27.6 ms, gradient 55.6 ms,
// with 32, 64 and 128 MiB alike).
// SHGO_ESP_SCRATCH_DOUBLES sets another size.
constexpr int64_t kPieceWords = (int64_t)1 << 23;

template <int NC>
cudaError_t launch_pieces(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work, int64_t nbf,
                          const double* D, int64_t npoints, const double* points, double* phi, cudaStream_t stream) {
  const Tables& th = tables_host();
  cudaStream_t* pool = nullptr;
  int npool = 0;
  cudaError_t e = pool_streams(&pool, &npool);
  if (e != cudaSuccess) return e;
  // classes by decreasing cost, dealt round-robin over the pool streams; each stream has one region of weights
  std::vector<int> order;
  for (size_t c = 0; c < work.size(); ++c)
    if (work[c].npairs > 0) order.push_back((int)c);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    auto cost = [&](int c) {
      const int lam = work[c].la + work[c].lb;
      return (double)work[c].npp * ((double)npoints * (lam + 3) * (lam + 3) + 20.0 * n_r(lam));
    };
    return cost(x) > cost(y);
  });
  const int ns = (int)std::min<size_t>(order.size(), (size_t)std::max(npool, 1));
  if (ns == 0) return cudaSuccess;
  int64_t words = kPieceWords;
  if (const char* env = std::getenv("SHGO_ESP_SCRATCH_DOUBLES")) words = std::max<int64_t>(1, std::atoll(env));
  std::vector<std::vector<ClassWork>> cut(order.size());
  std::vector<int64_t> at(ns, 0);
  int2* buf = nullptr;
  for (;; words /= 2) {  // smaller pieces where the device has no room for these, down to a shell pair at a time
    std::vector<int64_t> region(ns, 0);
    bool more = false;  // some piece has several shell pairs
    for (size_t k = 0; k < order.size(); ++k) {
      const ClassWork& w = work[order[k]];
      const int64_t per = weight_words(w.la + w.lb + (NC == 3), NC);
      cut[k] = pieces(w, db.h_ppoff, per, words);
      for (const ClassWork& c : cut[k]) {
        region[k % ns] = std::max(region[k % ns], c.npp * per);
        more |= c.npairs > 1;
      }
    }
    int64_t total = 0;
    for (int i = 0; i < ns; ++i) {
      at[i] = total;
      total += region[i];
    }
    e = workspace_alloc((void**)&buf, sizeof(int2) * (size_t)std::max<int64_t>(total, 1), stream);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || !more) return e;
  }
  cudaEvent_t fork = nullptr;
  e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(fork, stream);
  for (int i = 0; i < ns && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(pool[i], fork, 0);
  for (size_t k = 0; k < order.size() && e == cudaSuccess; ++k) {
    cudaStream_t s = pool[k % ns];
    for (const ClassWork& w : cut[k]) {
      const int lam = w.la + w.lb, lam1 = lam + (NC == 3), cid = class_id(w.la, w.lb);
      AdjointArgs a;
      a.la = w.la;
      a.lb = w.lb;
      a.npairs = w.npairs;
      a.pair_base = w.pair_base;
      a.pp_base = w.pp_base;
      a.pair_a = db.pair_a;
      a.pair_b = db.pair_b;
      a.pair_ppoff = db.pair_ppoff;
      a.pair_site = db.pair_site;
      a.rot_per = rot_block(db.rot_lmax);
      a.rotd = db.rotd;
      a.site_rot = db.site_rot;
      a.shell_nprim = db.shell_nprim;
      a.shell_foff = db.shell_foff;
      a.etab = dt.etab;
      a.eoff = dt.eoff;
      a.gt_ptr = dt.gt_ptr + th.gt_base[cid];
      a.gt_terms = dt.gt_terms + th.gt_termbase[cid];
      a.dt_ptr = dt.dt_ptr + th.dt_base[lam];
      a.dt_terms = dt.dt_terms;
      a.fr_terms = dt.fr_terms;
      a.rmap = dt.rmap + th.rmap_off[lam1];
      a.rnorm = dt.rnorm + th.rmap_off[lam1];
      a.ppd = db.ppd;
      a.D = D;
      a.ld = nbf;
      a.weights = buf + at[k % ns];
      const int nW = (w.la + 1) * (w.la + 1) * (w.lb + 1) * (w.lb + 1);
      k_esp_adjoint<NC><<<grid_cap_sm(w.npairs, 16), nW >= 1024 ? 128 : (nW >= 256 ? 64 : 32), adjoint_smem<NC>(w.la, w.lb),
                         s>>>(a);
      e = cudaGetLastError();
      EspArgs g;
      g.npp = w.npp;
      g.pp_base = w.pp_base;
      g.pp_pair = db.pp_pair;
      g.pair_a = db.pair_a;
      g.shell_xyz = db.shell_xyz;
      g.site_rot = db.site_rot;
      g.pair_site = db.pair_site;
      g.ppd = db.ppd;
      g.weights = a.weights;
      g.npoints = npoints;
      g.points = points;
      g.phi = phi;
      if (e == cudaSuccess) e = boys_top_table(lam1, &g.boys_top);
      g.nchunks = (int)((npoints + kPts - 1) / kPts);
      g.nsplit = (int)std::max<int64_t>(1, std::min<int64_t>(w.npp, (int64_t)152 * 6 / g.nchunks));
      if (e == cudaSuccess) {
        esp_kernel_at<NC>(lam1, Lams{})<<<g.nchunks * g.nsplit, 32 * kEspWarps, esp_smem_at<NC>(lam1, Lams{}), s>>>(g);
        e = cudaGetLastError();
      }
      if (e != cudaSuccess) break;
    }
  }
  bool joined = true;
  for (int i = 0; i < ns && fork && joined; ++i) {
    cudaEvent_t join;
    if (cudaEventCreateWithFlags(&join, cudaEventDisableTiming) != cudaSuccess) {
      joined = false;
      break;
    }
    cudaEventRecord(join, pool[i]);
    cudaStreamWaitEvent(stream, join, 0);
    cudaEventDestroy(join);
  }
  if (fork) cudaEventDestroy(fork);
  if (!joined) {
    // `stream` does not wait for every pool stream: finish their work before the weights are returned
    for (int i = 0; i < ns; ++i) cudaStreamSynchronize(pool[i]);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaErrorUnknown;
  }
  cudaFreeAsync(buf, stream);
  return e;
}

}  // namespace

shgo_status launch_esp(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work, int64_t nbf,
                       const double* D, int64_t npoints, const double* points, double* phi, bool gradient,
                       cudaStream_t stream, std::string* err) {
  cudaError_t e =
      cudaMemsetAsync(phi, 0, sizeof(double) * (size_t)std::max<int64_t>(npoints, 1) * (gradient ? 3 : 1), stream);
  if (e == cudaSuccess)
    e = gradient ? launch_pieces<3>(db, dt, work, nbf, D, npoints, points, phi, stream)
                 : launch_pieces<1>(db, dt, work, nbf, D, npoints, points, phi, stream);
  if (e != cudaSuccess) {
    *err = std::string("electrostatic potential: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? SHGO_ERR_OOM : SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}

cudaError_t esp_fp64_setup() {
  cudaError_t e = upload_nucleus_constants();
  if (e == cudaSuccess) e = set_max_dynamic_smem((const void*)k_esp_adjoint<1>);
  if (e == cudaSuccess) e = set_max_dynamic_smem((const void*)k_esp_adjoint<3>);
  for (int lam = 0; lam <= kLamMax && e == cudaSuccess; ++lam) {
    e = set_max_dynamic_smem((const void*)esp_kernel_at<1>(lam, Lams{}));
    if (e == cudaSuccess) e = set_max_dynamic_smem((const void*)esp_kernel_at<3>(lam + 1, Lams{}));
  }
  return e;
}

}  // namespace shgo
