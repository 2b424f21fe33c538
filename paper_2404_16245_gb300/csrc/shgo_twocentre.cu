// Matrices over shell pairs that depend on the vector between the two centres alone: overlap (Eqs. 9-10) and two-centre
// Coulomb integrals (a|b).  Both have blocks
//   B[ma][mb] = sum_{L, M} G(la ma, lb mb; L M) X_L S_LM(n),  L = la - lb, la - lb + 2, ..., la + lb,
// n the unit vector between the centres and G the product-rule coefficients of solid harmonics; only the X_L differ.
//
// Coulomb: with Eq. 3 each primitive is N (2 alpha)^{-l} S_l(grad_A) exp(-alpha |r - A|^2), so for R = A - B
// (grad_B = -grad_R on functions of R)
//   (a|b) = c_a c_b (2 alpha)^{-la} (2 beta)^{-lb} (-1)^lb S_la(grad_R) S_lb(grad_R) g(|R|^2),
//   g(u) = 2 pi^{5/2} / (alpha beta sqrt(alpha + beta)) F_0(rho u),  rho = alpha beta / (alpha + beta),
// the Coulomb integral of two s Gaussians.  The product rule gives S_la S_lb = sum_{L,M} G |v|^{2k} S_LM with
// k = (la + lb - L)/2, Hobson's theorem S_LM(grad) f(u) = 2^L S_LM(R) f^{(L)}(u), and the Laplacian of S_LM(R) f(u) is
// S_LM(R) (4u f'' + (4L + 6) f'), so X_L = 2^L (-|R|)^L sum_j a_{k,j}(L) u^j g^{(L+k+j)}(u), with
// g^{(n)}(u) = 2 pi^{5/2} / (alpha beta sqrt(alpha + beta)) (-rho)^n F_n(rho u), summed over primitive pairs.
//
// Overlap: both orbitals translated to P (Eq. 7) in the pair frame, where the one-centre integrals are diagonal,
//   int S_{l1 m1}(r_P) S_{l2 m2}(r_P) e^{-p r_P^2} = delta delta 4 pi (pi/2)^{1/2} (2 l1 - 1)!! / (2p)^{l1+3/2},
// so the block is diagonal there with d(m) = sum_{l1 >= m} K(m, l1) w(l1), and as S_LM(z) = delta_M0 the X_L solve
// sum_L G(la m, lb m; L 0) X_L = d(m), m = 0..lb: a (lb + 1)^2 system per class, inverted on the host (its condition is
// below 2.6 for every class to (8, 8)).
//
// What bounds it: FP64 at 1.7 lanes per clock and SM.  The scalar steps (Boys values, powers, divisions) therefore run
// with full lanes, one thread per primitive pair (Coulomb) or shell pair (overlap), in a launch of their own; the
// harmonics once per pair of centres; a warp per shell pair is left with one product per (L, M) and one multiply-add per
// coupling coefficient, about five per element.
//
// Measured (GB300, 32 atoms with l <= 6, 25,200 shell pairs): (a|b) 421 -> 63 us against one block per shell pair for all
// steps, overlap 95 -> 55 us against a warp per pair with D^la diag(d) (D^lb)^T.  Of that, rows of terms read coalesced
// instead of one list per lane and the harmonics in the radial launch instead of their own: 86 -> 63, 78 -> 55 us.  The overlap of small bases keeps
// the warp-per-pair form in one launch (overlap_in_one_launch).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <string>
#include <vector>

#include "shgo_internal.h"
#include "shgo_math.h"

namespace shgo {

namespace {

__constant__ HarmCoef k_harm;
__constant__ BoysConst k_boys;
// Per class: K(m, l1) cf(l1) at (m, l1) of a (lb + 1)^2 square (zero below m), then the inverse of G(la m, lb m; L 0) at
// (j, m), L = la + lb - 2 j; cf(l1) = 4 pi (pi/2)^{1/2} (2 l1 - 1)!! / 2^{l1 + 3/2}.
constexpr int kOvStride = 2 * (kLmax + 1) * (kLmax + 1);
__device__ double g_overlap[kNumClasses * kOvStride];

constexpr int kMaxClasses = kNumClasses;
struct PairClasses {  // classes with pairs: class c holds the items [first[c], first[c + 1])
  int n;
  int first[kMaxClasses + 1];
  int pair_base[kMaxClasses];
  int rows[kMaxClasses], terms[kMaxClasses];  // the class's coupling rows and terms (Tables::cx_base)
  unsigned char la[kMaxClasses], lb[kMaxClasses];
};

__device__ __forceinline__ int class_of_item(const PairClasses& cls, int item) {
  int c = 0, hi = cls.n - 1;
  while (c < hi) {
    const int mid = (c + hi + 1) >> 1;
    if (cls.first[mid] <= item)
      c = mid;
    else
      hi = mid - 1;
  }
  return c;
}

// Column M of S_LM(n), L = |M| .. lam, of the unit vector n = (B - A)/|B - A| (z for A = B): put(L, S_LM).
template <typename Put>
__device__ __forceinline__ void site_column(const double* __restrict__ n, int lam, int m, Put&& put) {
  const int am = m < 0 ? -m : m;
  const double x = n[0], y = n[1], z = n[2];
  double sp = 1.0, sm = 0.0;  // S_{l,l}, S_{l,-l}
  if (am >= 1) {
    sp = x;
    sm = y;
    for (int l = 1; l < am; ++l) {
      const double c = k_harm.c[l];
      const double np = c * (x * sp - y * sm), nm = c * (y * sp + x * sm);
      sp = np;
      sm = nm;
    }
  }
  double prv = 0.0, cur = m < 0 ? sm : sp;
  put(am, cur);
  for (int l = am; l < lam; ++l) {
    const int k = l * l + l + m;
    double v = k_harm.a[k] * (z * cur);
    if (m > -l && m < l) v -= k_harm.b[k] * prv;
    put(l + 1, v);
    prv = cur;
    cur = v;
  }
}

// The columns of every ordered pair of centres, one thread per column: the share of block `block` of `blocks`.  The radial
// launches carry these blocks after their own.
struct SiteArgs {
  int n_sites, lam;
  const double* site_rot;
  double* S;
};
__device__ __forceinline__ void site_harmonics(const SiteArgs& A, int block, int blocks) {
  const int lam = A.lam, ncol = 2 * lam + 1, ns = (lam + 1) * (lam + 1);
  for (int64_t t = block * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)A.n_sites * ncol;
       t += (int64_t)blocks * blockDim.x) {
    const int64_t site = t / ncol;
    const int m = (int)(t - site * ncol) - lam;
    double* o = A.S + site * ns;
    site_column(A.site_rot + 9 * site + 6, lam, m, [&](int l, double v) { o[l * l + l + m] = v; });
  }
}

// Coulomb: X of one primitive pair per thread, X[(q - q0) stride + k], L = la + lb - 2k.
__global__ void __launch_bounds__(128) k_coulomb_radial(int own, SiteArgs sites, int64_t q0, int64_t n, int stride, const int* __restrict__ pp_pair,
                                                        const int* __restrict__ pp_ij, const int* __restrict__ pair_a,
                                                        const int* __restrict__ pair_b,
                                                        const double* __restrict__ shell_xyz,
                                                        const int* __restrict__ shell_l,
                                                        const int* __restrict__ shell_poff,
                                                        const double* __restrict__ prim_exp,
                                                        const double* __restrict__ prim_coef,
                                                        const double* __restrict__ boys_tab,
                                                        const double* __restrict__ c2_a, double* __restrict__ X) {
  if (blockIdx.x >= own) {
    site_harmonics(sites, blockIdx.x - own, gridDim.x - own);
    return;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)own * blockDim.x) {
    const int pr = pp_pair[q0 + i], ij = pp_ij[q0 + i], a = pair_a[pr], b = pair_b[pr];
    const int la = shell_l[a], lb = shell_l[b], lam = la + lb;
    const int ia = shell_poff[a] + (ij >> 8), ib = shell_poff[b] + (ij & 255);
    const double al = prim_exp[ia], be = prim_exp[ib];
    const double Rx = shell_xyz[3 * a] - shell_xyz[3 * b], Ry = shell_xyz[3 * a + 1] - shell_xyz[3 * b + 1],
                 Rz = shell_xyz[3 * a + 2] - shell_xyz[3 * b + 2];
    const double u = Rx * Rx + Ry * Ry + Rz * Rz, r = sqrt(u);
    const double rp = 1.0 / (al + be), ra = 1.0 / al, rb = 1.0 / be, rho = al * be * rp;
    double v = prim_coef[ia] * prim_coef[ib] * 34.986836655249725693 * (ra * rb * sqrt(rp));  // 2 pi^{5/2}
    for (int k = 0; k < la; ++k) v *= 0.5 * ra;
    for (int k = 0; k < lb; ++k) v *= 0.5 * rb;
    double H[kLamMax + 1];
    boys_eval(lam, rho * u, H, 1, boys_tab, k_boys);
    double f = (lb & 1) ? -v : v;  // v (-rho)^n (-1)^lb
    for (int k = 0; k <= lam; ++k) {
      H[k] *= f;
      f *= -rho;
    }
    double rl = 1.0;  // (-2 |R|)^L from the lowest L up
    for (int k = 0; k < la - lb; ++k) rl *= -2.0 * r;
    double* o = X + i * stride;
    for (int k = lb; k >= 0; --k) {
      const int L = lam - 2 * k;
      const double* ak = c2_a + ((size_t)L * (kC2K + 1) + k) * (kC2K + 1);
      double s = 0.0, uj = 1.0;
      for (int j = 0; j <= k; ++j) {
        s = fma(ak[j] * uj, H[L + k + j], s);
        uj *= u;
      }
      o[k] = s * rl;
      rl *= 4.0 * u;
    }
  }
}

// Overlap: X of one shell pair per thread, X[item stride + j], L = la + lb - 2j.
__global__ void __launch_bounds__(128) k_overlap_radial(int own, SiteArgs sites, PairClasses cls, int stride, const int* __restrict__ pair_a,
                                                        const int* __restrict__ pair_b,
                                                        const int64_t* __restrict__ pair_ppoff,
                                                        const int* __restrict__ pair_site, int64_t rot_per,
                                                        const double* __restrict__ rotd,
                                                        const int* __restrict__ shell_nprim,
                                                        const PPData* __restrict__ ppd, double* __restrict__ X) {
  if (blockIdx.x >= own) {
    site_harmonics(sites, blockIdx.x - own, gridDim.x - own);
    return;
  }
  const int total = cls.first[cls.n];
  for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < total; item += own * blockDim.x) {
    const int c = class_of_item(cls, item), la = cls.la[c], lb = cls.lb[c];
    const int pr = cls.pair_base[c] + (item - cls.first[c]);
    const int npp = shell_nprim[pair_a[pr]] * shell_nprim[pair_b[pr]];
    const double r = rotd[(int64_t)pair_site[pr] * rot_per];
    double w[kLmax + 1];
    for (int k = 0; k <= lb; ++k) w[k] = 0.0;
    const PPData* pp = ppd + pair_ppoff[pr];
    for (int i = 0; i < npp; ++i) {
      const PPData pd = pp[i];
      if (pd.pref == 0.0) continue;
      // w(lb) = pref p^{-3/2} (beta/p)^{la-lb} p^{-lb}, w(l1 - 1) = w(l1) p (beta/p)(alpha/p)
      double v = pd.pref * pd.rp * (pd.sp * pd.rp);
      for (int k = 0; k < la - lb; ++k) v *= pd.ra;
      for (int k = 0; k < lb; ++k) v *= pd.rp;
      const double f = pd.ra * pd.rb * pd.p;
      for (int l1 = lb; l1 >= 0; --l1) {
        w[l1] += v;
        v *= f;
      }
    }
    // |b - a|^{la - l1} (-|b - a|)^{lb - l1}
    double rl = 1.0;
    for (int k = 0; k < la - lb; ++k) rl *= r;
    for (int l1 = lb; l1 >= 0; --l1) {
      w[l1] *= rl;
      rl *= -(r * r);
    }
    const double* K = g_overlap + (size_t)(la * (la + 1) / 2 + lb) * kOvStride;
    const double* Ti = K + (kLmax + 1) * (kLmax + 1);
    double x[kLmax + 1];
    for (int j = 0; j <= lb; ++j) x[j] = 0.0;
    for (int m = 0; m <= lb; ++m) {
      double d = 0.0;
      for (int l1 = m; l1 <= lb; ++l1) d = fma(K[m * (lb + 1) + l1], w[l1], d);
      for (int j = 0; j <= lb; ++j) x[j] = fma(Ti[j * (lb + 1) + m], d, x[j]);
    }
    for (int j = 0; j <= lb; ++j) X[(int64_t)item * stride + j] = x[j];
  }
}

// Blocks from the X_L: a warp per shell pair, four per block.  nx[] = rows of X per pair: its primitive pairs from
// pair_ppoff - q0 on (Coulomb), or the item itself (per_pair).  S: the harmonics of every pair of centres, or NULL, and the
// warp forms those of its pair.
constexpr int kBlockWarps = 4;
__global__ void __launch_bounds__(32 * kBlockWarps) k_twocentre_blocks(
    PairClasses cls, int lam_max, int stride, bool per_pair, int64_t q0, const int* __restrict__ pair_a,
    const int* __restrict__ pair_b, const int64_t* __restrict__ pair_ppoff, const int* __restrict__ pair_site,
    const double* __restrict__ site_rot, const int* __restrict__ shell_nprim, const int64_t* __restrict__ shell_foff,
    const double* __restrict__ S, const double* __restrict__ X, const int2* __restrict__ cx_rows, const GTerm* __restrict__ cx_terms, MolView mv,
    double* __restrict__ out) {
  extern __shared__ double smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, ns = (lam_max + 1) * (lam_max + 1);
  double* SX = smem + wib * (ns + kLmax + 1);  // [ns] X_L S_LM(n)
  double* xs = SX + ns;
  const int total = cls.first[cls.n];
  for (int item = blockIdx.x * kBlockWarps + wib; item < total; item += gridDim.x * kBlockWarps) {
    const int c = class_of_item(cls, item), la = cls.la[c], lb = cls.lb[c], lam = la + lb;
    const int pr = cls.pair_base[c] + (item - cls.first[c]);
    const int a = pair_a[pr], b = pair_b[pr];
    const int nx = per_pair ? 1 : shell_nprim[a] * shell_nprim[b];
    const double* x0 = X + (per_pair ? (int64_t)item : pair_ppoff[pr] - q0) * stride;
    __syncwarp();  // the warp's previous pair is done with its tables
    if (lane <= lb) {
      double s = 0.0;
      for (int i = 0; i < nx; ++i) s += x0[(int64_t)i * stride + lane];
      xs[lane] = s;
    }
    __syncwarp();
    if (S) {
      const double* Sp = S + (int64_t)pair_site[pr] * ns;
      for (int k = 0; k <= lb; ++k) {
        const int L = lam - 2 * k;
        const double x = xs[k];
        for (int m = lane; m <= 2 * L; m += 32) SX[L * L + m] = Sp[L * L + m] * x;
      }
    } else {
      for (int m = lane - lam; m <= lam; m += 32)
        site_column(site_rot + 9 * (int64_t)pair_site[pr] + 6, lam, m, [&](int l, double v) {
          if (l >= la - lb && ((lam - l) & 1) == 0) SX[l * l + l + m] = v * xs[(lam - l) >> 1];
        });
    }
    __syncwarp();
    const int2* rows = cx_rows + cls.rows[c];
    const GTerm* terms = cx_terms + cls.terms[c];
    const int na = 2 * la + 1, nb = 2 * lb + 1;
    const int64_t fa0 = shell_foff[a], fb0 = shell_foff[b];
    int64_t obase, ld;
    mol_output(mv, pr, obase, ld);
    double* o = out + obase;
    // a diagonal block's entries (ma, mb) and (mb, ma) have equal lists: exactly symmetric
    for (int r = lane; r < ((na * nb + 31) & ~31); r += 32) {
      const int2 row = __ldg(rows + r);
      const int K = row.x >> 16, e = row.x & 0xffff;
      const GTerm* tp = terms + row.y;
      double v = 0.0;
#pragma unroll 4
      for (int j = 0; j < K; ++j) {
        const GTerm g = tp[32 * j];
        v = fma(g.coef, SX[g.ridx], v);
      }
      if (e != 0xffff) {
        const int ma = e / nb, mb = e - ma * nb;
        o[(fa0 + ma) * ld + fb0 + mb] = v;
        if (a != b) o[(fb0 + mb) * ld + fa0 + ma] = v;
      }
    }
  }
}

// Overlap of small bases, all steps of a shell pair in one warp and one launch: S' = diag(d) of the pair frame rotated
// back, S = D^{la} diag(d) (D^{lb})^T.  More FP64 operations than the X_L form but no second launch, no tables and no
// work array in between (rule and figures at overlap_in_one_launch).
//
// Shared doubles of one warp for angular momenta up to lm: D^{la} and D^{lb}, t_A and t_B, w(l1), |b - a|^k,
// d(m) and X = D^{la} diag(d).
__host__ __device__ inline int overlap_warp_doubles(int lm) {
  const int n = 2 * lm + 1;
  return 3 * n * n + 2 * (lm + 1) * n + 2 * (lm + 1) + n + 1;
}

__global__ void __launch_bounds__(32 * kBlockWarps) k_overlap(PairClasses cls, int lm_max,
                                                                const int* __restrict__ pair_a,
                                                                const int* __restrict__ pair_b,
                                                                const int64_t* __restrict__ pair_ppoff,
                                                                const int* __restrict__ pair_site, int64_t rot_per,
                                                                const double* __restrict__ rotd,
                                                                const int* __restrict__ shell_nprim,
                                                                const int64_t* __restrict__ shell_foff,
                                                                const double* __restrict__ etab,
                                                                const int* __restrict__ eoff,
                                                                const PPData* __restrict__ ppd, MolView mv,
                                                                double* __restrict__ out) {
  extern __shared__ double smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  double* wsm = smem + wib * overlap_warp_doubles(lm_max);
  const int total = cls.first[cls.n];
  for (int item = blockIdx.x * kBlockWarps + wib; item < total; item += gridDim.x * kBlockWarps) {
    const int c = class_of_item(cls, item);
    const int la = cls.la[c], lb = cls.lb[c];
    const int pr = cls.pair_base[c] + (item - cls.first[c]);
    const int na = 2 * la + 1, nb = 2 * lb + 1;
    const int lm = la > lb ? la : lb, ln = la < lb ? la : lb;
    const int nDb = la != lb ? nb * nb : 0;
    double* Dm = wsm;  // D^{la}(Q^T), then D^{lb}(Q^T) when lb != la
    double* tA = Dm + na * na + nb * nb;
    double* tB = tA + (la + 1) * na;
    double* wl = tB + (lb + 1) * nb;  // w(l1)
    double* dpow = wl + lm + 1;       // |b - a|^k
    double* dm = dpow + lm + 1;       // d(m), m = -ln..ln
    double* X = dm + 2 * lm + 1;      // [ma][m] = D^{la}[ma][m] d(m)
    const int nm = 2 * ln + 1;
    const int a = pair_a[pr], b = pair_b[pr];
    const double* rd = rotd + (int64_t)pair_site[pr] * rot_per;
    __syncwarp();  // the warp's previous pair is done with its tables
    if (lane == 0) {
      const double dist = rd[0];
      double v = 1.0;
      for (int k = 0; k <= lm; ++k) {
        dpow[k] = v;
        v *= dist;
      }
    }
    for (int e = lane; e < na * na; e += 32) Dm[e] = rd[1 + rot_doff(la) + e];
    for (int e = lane; e < nDb; e += 32) Dm[na * na + e] = rd[1 + rot_doff(lb) + e];
    // radial sums over primitive pairs, one l1 per lane
    if (lane <= ln) {
      const int l1 = lane;
      double dfact = 1.0;
      for (int k = 2 * l1 - 1; k > 1; k -= 2) dfact *= k;
      // 4 pi (pi/2)^{1/2} / 2^{l1 + 3/2} (2 l1 - 1)!!
      double cf = 4.0 * 3.14159265358979323846 * 1.2533141373155002512 * dfact * 0.35355339059327376220;
      for (int k = 0; k < l1; ++k) cf *= 0.5;
      const int64_t q0 = pair_ppoff[pr];
      const int npp = shell_nprim[a] * shell_nprim[b];
      double acc = 0.0;
      for (int ij = 0; ij < npp; ++ij) {
        const PPData pd = ppd[q0 + ij];
        if (pd.pref == 0.0) continue;
        double v = pd.pref * pd.rp * (pd.sp * pd.rp);  // p^{-3/2}
        for (int k = 0; k < l1; ++k) v *= pd.rp;
        for (int k = 0; k < la - l1; ++k) v *= pd.ra;
        for (int k = 0; k < lb - l1; ++k) v *= pd.rb;
        acc += v;
      }
      wl[l1] = cf * acc;
    }
    __syncwarp();
    for (int e = lane; e < (la + 1) * na; e += 32) {
      const int l1 = e / na, ma = e % na - la, lr = la - l1;
      tA[e] = l1 >= (ma < 0 ? -ma : ma) ? etab[eoff[la] + translation_offset_dev(la, ma, l1, ma) + lr] * dpow[lr] : 0.0;
    }
    for (int e = lane; e < (lb + 1) * nb; e += 32) {
      const int l2 = e / nb, mb = e % nb - lb, lr = lb - l2;
      tB[e] = l2 >= (mb < 0 ? -mb : mb)
                  ? etab[eoff[lb] + translation_offset_dev(lb, mb, l2, mb) + lr] * ((lr & 1) ? -dpow[lr] : dpow[lr])
                  : 0.0;
    }
    __syncwarp();
    // S' = diag(d), d(m) = sum_{l1 >= |m|} t_A(l1, m) t_B(l1, m) w(l1) for |m| <= min(la, lb), once per pair
    if (lane < nm) {
      const int m = lane - ln, am = m < 0 ? -m : m;
      double d = 0.0;
      for (int l1 = am; l1 <= ln; ++l1) d = fma(tA[l1 * na + m + la] * tB[l1 * nb + m + lb], wl[l1], d);
      dm[lane] = d;
    }
    __syncwarp();
    const double* Da = Dm;
    const double* Db = la != lb ? Dm + na * na : Dm;
    for (int e = lane; e < na * nm; e += 32) {
      const int r = e / nm, j = e - r * nm;
      X[e] = Da[r * na + j - ln + la] * dm[j];
    }
    __syncwarp();
    // S = X (D^{lb})^T; a diagonal block (a == b) takes the entry below its diagonal from the products of the
    // entry above it, so it is exactly symmetric
    const int64_t fa0 = shell_foff[a], fb0 = shell_foff[b];
    int64_t obase, ld;
    mol_output(mv, pr, obase, ld);
    double* o = out + obase;
    for (int e = lane; e < na * nb; e += 32) {
      const int ma = e / nb, mb = e % nb;
      const bool lower = a == b && ma > mb;
      const int r = lower ? mb : ma, q = lower ? ma : mb;
      double s = 0.0;
      for (int j = 0; j < nm; ++j) s = fma(X[r * nm + j], Db[q * nb + j - ln + lb], s);
      o[(fa0 + ma) * ld + fb0 + mb] = s;
      if (a != b) o[(fb0 + mb) * ld + fa0 + ma] = s;
    }
  }
}

// FP64 warp instructions of k_overlap for the shell pairs of `work`, about: per primitive pair the power products, per shell
// pair the translation factors and the rotation.  Up to kOneLaunch of them per SM (FP64 takes 19 clocks each) the one
// launch is over before the two launches of the X_L form, whose chains take 20 to 90 us whatever the size.  Measured (GB300,
// one launch and two, with the count per SM): 2 atoms with l <= 8 (100) 23 and 47 us, 10 with l <= 3 contracted (1000) 17 and
// 32, 3 contracted atoms up to g shells (1400) 59 and 92, 40 with l <= 2 (2200) 17 and 26, 14 with l <= 6 (2300) 25 and 32,
// 16 with l <= 6 (3000) 34 and 31, 20 with l <= 6 (4600) 41 and 36.
constexpr int64_t kOneLaunch = 2600;
bool overlap_in_one_launch(const std::vector<ClassWork>& work) {
  int64_t w = 0;
  for (const ClassWork& c : work) {
    const int na = 2 * c.la + 1, nb = 2 * c.lb + 1;
    const auto rows = [](int n) { return (n + 31) / 32; };
    w += c.npp * (14 + c.la + c.lb) + c.npairs * (int64_t)(20 + c.la + 3 * c.lb + rows(na * nb) * (nb + 2) +
                                                          rows((c.la + 1) * na) + rows((c.lb + 1) * nb));
  }
  return w <= kOneLaunch * grid_cap_sm(INT64_MAX, 1);
}

shgo_status launch_overlap_small(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work,
                                 const MolView& mv, double* out, cudaStream_t stream, std::string* err) {
  PairClasses cls{};
  int total = 0, lm = 0;
  for (const ClassWork& w : work) {
    if (w.npairs == 0) continue;
    cls.first[cls.n] = total;
    cls.pair_base[cls.n] = w.pair_base;
    cls.la[cls.n] = (unsigned char)w.la;
    cls.lb[cls.n] = (unsigned char)w.lb;
    ++cls.n;
    total += w.npairs;
    lm = std::max(lm, w.la);
  }
  cls.first[cls.n] = total;
  if (total == 0) return SHGO_OK;
  k_overlap<<<grid_cap_sm(((int64_t)total + kBlockWarps - 1) / kBlockWarps, 12), 32 * kBlockWarps,
              sizeof(double) * kBlockWarps * (size_t)overlap_warp_doubles(lm), stream>>>(
      cls, lm, db.pair_a, db.pair_b, db.pair_ppoff, db.pair_site, rot_block(db.rot_lmax), db.rotd, db.shell_nprim,
      db.shell_foff, dt.etab, dt.eoff, db.ppd, mv, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    *err = std::string("overlap launch: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}

// Doubles of X formed at a time (128 MiB); larger bases run in pieces of whole shell pairs.  S is formed whole: it takes
// (2 lmax + 1)^2 doubles per pair of centres, no more than the matrix where centres carry shells of the basis's lmax.  Where
// the device has no room for it each warp forms the harmonics of its pair (300 atoms with l <= 3: overlap 0.60 -> 1.76 ms,
// (a|b) 0.80 -> 1.97 ms).  SHGO_TWOCENTRE_SCRATCH_DOUBLES sets another size of X, and a limit for S.
constexpr int64_t kXDoubles = (int64_t)1 << 24;

shgo_status launch_twocentre(bool coulomb, const DeviceBasis& db, const DeviceTables& dt,
                             const std::vector<ClassWork>& work, const MolView& mv, double* out, cudaStream_t stream,
                             std::string* err) {
  const int lam_max = 2 * db.rot_lmax, stride = db.rot_lmax + 1, ns = (lam_max + 1) * (lam_max + 1);
  int64_t npairs = 0, npp = 0;
  for (const ClassWork& w : work) {
    npairs += w.npairs;
    npp += w.npp;
  }
  if (npairs == 0) return SHGO_OK;
  int64_t xcap = kXDoubles, scap = INT64_MAX;
  if (const char* env = std::getenv("SHGO_TWOCENTRE_SCRATCH_DOUBLES")) xcap = scap = std::max<int64_t>(1, std::atoll(env));
  int64_t slen = (int64_t)db.n_sites * ns <= scap ? (int64_t)db.n_sites * ns : 0;
  std::vector<std::vector<ClassWork>> pieces;
  double* buf = nullptr;  // S of every pair of centres, then X
  for (;;) {  // less at a time where the device has no room: no S, then smaller pieces, down to a shell pair
    // pieces: consecutive (class, pairs) runs whose rows of X fit
    pieces.assign(1, {});
    int64_t rows = 0, most = 0;
    for (const ClassWork& w : work) {
      for (int q = w.pair_base; q < w.pair_base + w.npairs;) {
        ClassWork c{w.la, w.lb, 0, q, 0, db.h_ppoff[q]};
        int64_t r = 0;
        while (q < w.pair_base + w.npairs) {
          const int64_t add = coulomb ? db.h_ppoff[q + 1] - db.h_ppoff[q] : 1;
          if (rows + r + add > std::max<int64_t>(xcap / stride, 1) && rows + r > 0) break;
          r += add;
          ++c.npairs;
          ++q;
        }
        c.npp = db.h_ppoff[q] - c.pp_base;
        if (c.npairs) pieces.back().push_back(c);
        rows += r;
        most = std::max(most, rows);
        if (q < w.pair_base + w.npairs) {
          pieces.emplace_back();
          rows = 0;
        }
      }
    }
    const cudaError_t e = workspace_alloc((void**)&buf, sizeof(double) * (size_t)(slen + most * stride), stream);
    if (e == cudaSuccess) break;
    cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || (slen == 0 && xcap <= stride)) {
      *err = std::string("two-centre buffers: ") + cudaGetErrorString(e);
      return SHGO_ERR_OOM;
    }
    if (slen > 0)
      slen = 0;
    else
      xcap = std::min(xcap, most * stride) / 2;
  }
  double *S = slen > 0 ? buf : nullptr, *X = buf + slen;
  const Tables& th = tables_host();
  const int site_blocks = S ? grid_cap_sm(((int64_t)db.n_sites * (2 * lam_max + 1) + 127) / 128, 16) : 0;
  const SiteArgs sites{db.n_sites, lam_max, db.site_rot, S};
  bool first = true;
  for (const std::vector<ClassWork>& piece : pieces) {
    if (piece.empty()) continue;
    PairClasses cls{};
    int total = 0;
    int64_t pp = 0;
    for (const ClassWork& w : piece) {
      cls.first[cls.n] = total;
      cls.pair_base[cls.n] = w.pair_base;
      cls.la[cls.n] = (unsigned char)w.la;
      cls.lb[cls.n] = (unsigned char)w.lb;
      cls.rows[cls.n] = th.cx_base[2 * class_id(w.la, w.lb)];
      cls.terms[cls.n] = th.cx_base[2 * class_id(w.la, w.lb) + 1];
      ++cls.n;
      total += w.npairs;
      pp += w.npp;
    }
    cls.first[cls.n] = total;
    const int64_t q0 = piece[0].pp_base;
    const int own = grid_cap_sm(((coulomb ? pp : (int64_t)total) + 127) / 128, 16), more = first ? site_blocks : 0;
    first = false;
    if (coulomb)
      k_coulomb_radial<<<own + more, 128, 0, stream>>>(own, sites, q0, pp, stride, db.pp_pair, db.pp_ij, db.pair_a, db.pair_b,
                                                       db.shell_xyz, db.shell_l, db.shell_poff, db.prim_exp, db.prim_coef,
                                                       dt.boys, dt.c2_a, X);
    else
      k_overlap_radial<<<own + more, 128, 0, stream>>>(own, sites, cls, stride, db.pair_a, db.pair_b, db.pair_ppoff,
                                                       db.pair_site, rot_block(db.rot_lmax), db.rotd, db.shell_nprim, db.ppd,
                                                       X);
    k_twocentre_blocks<<<grid_cap_sm(((int64_t)total + kBlockWarps - 1) / kBlockWarps, 12), 32 * kBlockWarps,
                         sizeof(double) * kBlockWarps * (size_t)(ns + kLmax + 1), stream>>>(
        cls, lam_max, stride, !coulomb, q0, db.pair_a, db.pair_b, db.pair_ppoff, db.pair_site, db.site_rot,
        db.shell_nprim, db.shell_foff, S, X, dt.cx_rows, dt.cx_terms, mv, out);
  }
  const cudaError_t e = cudaGetLastError();
  cudaFreeAsync(buf, stream);
  if (e != cudaSuccess) {
    *err = std::string(coulomb ? "two-centre launch: " : "overlap launch: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}

}  // namespace

shgo_status launch_overlap(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work,
                           const MolView& mv, double* out, cudaStream_t stream, std::string* err) {
  if (overlap_in_one_launch(work)) return launch_overlap_small(db, dt, work, mv, out, stream, err);
  return launch_twocentre(false, db, dt, work, mv, out, stream, err);
}

shgo_status launch_coulomb2c(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work,
                             const MolView& mv, double* out, cudaStream_t stream, std::string* err) {
  return launch_twocentre(true, db, dt, work, mv, out, stream, err);
}

cudaError_t twocentre_setup() {
  std::vector<double> ov((size_t)kNumClasses * kOvStride, 0.0);
  for (int la = 0; la <= kLmax; ++la)
    for (int lb = 0; lb <= la; ++lb) {
      const int n = lb + 1;
      double* K = ov.data() + (size_t)class_id(la, lb) * kOvStride;
      double* Ti = K + (kLmax + 1) * (kLmax + 1);
      std::vector<long double> A((size_t)n * 2 * n, 0.0L);  // [G | 1], reduced to [1 | G^-1]
      for (int m = 0; m < n; ++m) {
        long double cf = 4.0L * 3.14159265358979323846264338328L * 1.25331413731550025120788264241L *
                         0.353553390593273762200422181052L;  // 4 pi (pi/2)^{1/2} 2^{-3/2}
        for (int l1 = 0; l1 < n; ++l1) {
          if (l1 > 0) cf *= (2 * l1 - 1) / 2.0L;
          if (l1 >= m)
            K[m * n + l1] = (double)((long double)translation_real(la, m, l1, m, 0) * translation_real(lb, m, l1, m, 0) * cf);
        }
        for (int j = 0; j < n; ++j) A[m * 2 * n + j] = gaunt_real(la, m, lb, m, la + lb - 2 * j, 0);
        A[m * 2 * n + n + m] = 1.0L;
      }
      for (int c = 0; c < n; ++c) {
        int p = c;
        for (int r = c + 1; r < n; ++r)
          if (std::fabs(A[r * 2 * n + c]) > std::fabs(A[p * 2 * n + c])) p = r;
        for (int k = 0; k < 2 * n; ++k) std::swap(A[c * 2 * n + k], A[p * 2 * n + k]);
        const long double d = A[c * 2 * n + c];
        for (int k = 0; k < 2 * n; ++k) A[c * 2 * n + k] /= d;
        for (int r = 0; r < n; ++r) {
          if (r == c) continue;
          const long double f = A[r * 2 * n + c];
          for (int k = 0; k < 2 * n; ++k) A[r * 2 * n + k] -= f * A[c * 2 * n + k];
        }
      }
      for (int j = 0; j < n; ++j)
        for (int m = 0; m < n; ++m) Ti[j * n + m] = (double)A[j * 2 * n + n + m];
    }
  cudaError_t e = cudaMemcpyToSymbol(g_overlap, ov.data(), sizeof(double) * ov.size());
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(k_harm, &harm_coef_host(), sizeof(HarmCoef));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(k_boys, &boys_const_host(), sizeof(BoysConst));
  return e;
}

}  // namespace shgo
