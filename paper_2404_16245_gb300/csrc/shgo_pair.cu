// Pair kernel (steps S3 to S5).
//
// Per shell pair, in the pair frame, the coupling blocks R'[L,M,k] of its primitive pairs are first contracted,
//   Rt[l1 l2][L M] = sum_ij f_ij(l1, l2) R'_ij[L, M, (l1 + l2 - L)/2],
//   f_ij = c_i c_j K_AB (beta/p)^{la-l1} (alpha/p)^{lb-l2}   (Eq. 11),
// so that the Clebsch-Gordan coupling runs once per shell pair instead of once per primitive pair:
//   W[l1 m1][l2 m2] = sum_{L,M} G(l1 m1, l2 m2; L M) Rt[l1 l2][L M],
//   Z[l1 m1][mb] = sum_{l2} t_B(l2, mb) W[l1 m1][l2 mb],   V' = t_A Z (both diagonal in m),
// then the rotation back and the write.
//
// What bounds it: in FP64 (1.7 lanes per clock and SM) the coupling is nearly half of the operations; integer
// multiply-adds issue at 62.  Rt is therefore held as 58-bit fixed point with one exponent per (l1, l2); the coupling
// coefficients are at most 1 and a row's absolute sum at most 1.33, so W stays in fixed point without a test, and the
// factors of Z are scaled per (l1, |mb|).  W is then within 2^-57 or so of the largest entry of its (l1, l2), Z of its
// largest product.  Rt, Z, V' and the rotation stay FP64.  The rest is latency: the threads take every entry of a chunk of eight primitive pairs without a
// barrier, and a row of the coupling program is one header and K coalesced 16-byte terms.
//
// Measured (GB300, pair phase of one V, against FP64 throughout with the coupling once per primitive pair): contracted
// 29-atom molecule 1.14 -> 0.37 ms (V 4.40 -> 3.79 ms, six such molecules 29.8 -> 27.6 ms); 32 atoms with l <= 6,
// uncontracted, 0.184 -> 0.160 ms (V 404 -> 392 us).  One scale per (l1, l2) for single primitive pairs too, instead of
// one per degree l1 + l2 over entries that (l1, l2) does not read: the same time (V of the 32 atoms 373 and 375 us), and
// blocks of high degrees alone, as on one centre with la - lb >= 2, keep their digits ((6, 2), p = 100, a nucleus 20 bohr off:
// 5.7e-8 of the largest element before).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "shgo_fixed.cuh"
#include "shgo_internal.h"

namespace shgo {

namespace {

constexpr int kChunk = 8;  // primitive pairs whose factors are tabulated at a time

// Shared memory, regions reused from phase to phase: W, later V' and its half-rotated form; the coupling entries, later
// the rotation matrices.
struct PairSmem {
  int wx, vp, yb, rt, dm, zb, ta, tb, pw, fab, cx, part;  // offsets in 8-byte words
  int en, ec, lo;                                         // offsets in ints after them
  int nints;
  size_t bytes;
};

__host__ __device__ inline int imax(int x, int y) { return x > y ? x : y; }

__host__ __device__ inline PairSmem pair_layout(int la, int lb, int nrt, int nth) {
  const int nWa = (la + 1) * (la + 1), na = 2 * la + 1, nb = 2 * lb + 1, nc = (la + 1) * (lb + 1) * (lb + 2) / 2;
  PairSmem s;
  s.wx = 0;
  s.vp = 0;
  s.yb = na * nb;
  int o = imax(nWa * w_stride(lb), 2 * na * nb);
  s.rt = s.dm = o;
  o += imax(nrt, na * na + nb * nb);
  s.pw = o;
  s.fab = o + kChunk * (la + lb + 2);
  o += kChunk * (la + lb + 2 + (la + 1) * (lb + 1));
  s.cx = o;
  o += nc;
  s.zb = o;
  o += nWa * nb;
  s.ta = o;
  o += (la + 1) * (la + 1);
  s.tb = o;
  o += (lb + 1) * (lb + 1);
  s.part = o;
  o += nrt < nth ? nth : 0;
  s.nints = 2 * o;
  s.en = 0;
  s.ec = (la + 1) * (lb + 1);
  s.lo = 2 * (la + 1) * (lb + 1);
  s.bytes = 8 * (size_t)o + 4 * (size_t)(s.lo + nWa);
  return s;
}

constexpr int kNoScale = -100000, kNotFinite = 1 << 20;

__global__ void __launch_bounds__(128) k_pair_block(PairArgs A) {
  extern __shared__ __align__(16) double smem[];
  __shared__ long long s_next[2];
  __shared__ unsigned long long s_t0;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int la = A.la, lb = A.lb, nR = n_r(la + lb), nrt = A.nrt;
  const int nWa = (la + 1) * (la + 1), nW = nWa * (lb + 1) * (lb + 1), nbk = (la + 1) * (lb + 1);
  const int ws = w_stride(lb), nrp = (nW + 31) & ~31;
  const int na = 2 * la + 1, nb = 2 * lb + 1, np = (lb + 1) * (lb + 2) / 2, nc = (la + 1) * np;
  const int nDb = la != lb ? nb * nb : 0;
  const PairSmem sm = pair_layout(la, lb, nrt, nth);
  int2* Wx = reinterpret_cast<int2*>(smem + sm.wx);  // [l1 m1][l2 m2], row stride ws
  double* Rt = smem + sm.rt;                          // contracted coupling entries, then their fixed point
  int2* Rx = reinterpret_cast<int2*>(Rt);
  double* Zb = smem + sm.zb;                          // [l1 m1][mb]
  double* Dm = smem + sm.dm;                          // D^{la}(Q^T), then D^{lb}(Q^T) when lb != la
  double* tA = smem + sm.ta;                          // [l1][|ma|]
  double* tB = smem + sm.tb;                          // [l2][|mb|]
  double* Vp = smem + sm.vp;                          // [ma][mb] in the pair frame, later the final block
  double* Yb = smem + sm.yb;
  double* pw = smem + sm.pw;                          // per primitive pair (beta/p)^k, k <= la, (alpha/p)^k, k <= lb
  double* fab = smem + sm.fab;                        // per primitive pair f(l1, l2)
  int2* cx = reinterpret_cast<int2*>(smem + sm.cx);   // [l1][l2, |mb|] t_B with the scale of (l1, l2), fixed point
  double* part = smem + sm.part;
  int* ints = reinterpret_cast<int*>(smem) + sm.nints;
  int* En = ints + sm.en;  // biased exponent of Rt per (l1, l2)
  int* Ec = ints + sm.ec;  // biased exponent of t_B times that scale per (l1, |mb|)
  int* lo = ints + sm.lo;  // l of a packed harmonic index
  for (int e = tid; e < nWa; e += nth) {
    int l = 0;
    while ((l + 1) * (l + 1) <= e) ++l;
    lo[e] = l;
  }
  // few entries: G groups of threads take every G-th primitive pair, their sums added in group order
  const float inv_nwa = 1.0f / (float)nWa;
  const int G = nrt < nth ? min(nth / nrt, kChunk) : 1;
  wq_for_each(A.wq, A.npairs, s_next, &s_t0, [&](long long wn) {
    const int pr = A.pair_base + (int)wn;
    const int a = A.pair_a[pr], b = A.pair_b[pr];
    const double* rd = A.rotd + (int64_t)A.pair_site[pr] * A.rot_per;
    const int npp = A.shell_nprim[a] * A.shell_nprim[b];
    const int64_t q0 = A.pair_ppoff[pr];
    const double dist = rd[0];
    // one primitive pair: the entries are R' itself, blocks (l1, l2) and (l2, l1) share them, and f joins the factors of Z.
    // A block's scale comes from the degrees L it reads alone: for far nuclei R' falls as t^{-(L+1)}, and a pair on one
    // centre has nothing but (la, lb), with L >= la - lb
    const bool single = npp == 1 && A.nrs < nrt;
    const auto scale_of = [&](int l1, int l2) {
      return single && l1 < l2 ? l2 * (lb + 1) + l1 : l1 * (lb + 1) + l2;
    };
    __syncthreads();  // the previous pair is done with the tables
    // translation along z (Eq. 7 with Eq. 8 coefficients, real basis): only nu = 0 survives,
    // t_A(l1, ma) = E^{la}(ma; l1 ma; 0) |b-a|^{la-l1}, t_B(l2, mb) = E^{lb}(mb; l2 mb; 0) (-|b-a|)^{lb-l2}; both depend on
    // |m| alone
    for (int e = tid; e < (la + 1) * (la + 1) + (lb + 1) * (lb + 1); e += nth) {
      const bool isb = e >= (la + 1) * (la + 1);
      const int l = isb ? lb : la, x = isb ? e - (la + 1) * (la + 1) : e, l1 = x / (l + 1);
      double v = __ldg(A.axial + l * (kLmax + 1) * (kLmax + 1) + x);  // 0 for l1 < |m|
      const double d = isb ? -dist : dist;
      for (int k = 0; k < l - l1; ++k) v *= d;
      (isb ? tB : tA)[x] = v;
    }
    for (int e = tid; e < nbk; e += nth) En[e] = 0;
    bool live = false;  // uniform over the block
    for (int i0 = 0; i0 < npp; i0 += kChunk) {
      const int n = min(kChunk, npp - i0);
      __syncthreads();  // the factors of the previous chunk are consumed
      // powers of beta/p and alpha/p, one per thread
      for (int x = tid; x < n * (la + lb + 2); x += nth) {
        const int i = x / (la + lb + 2), y = x - i * (la + lb + 2), k = y <= la ? y : y - la - 1;
        const PPData* pd = A.ppd + q0 + i0 + i;
        const double base = y <= la ? pd->ra : pd->rb;
        double v = y <= la ? pd->pref : 1.0;
        for (int j = 0; j < k; ++j) v *= base;
        pw[x] = v;
      }
      __syncthreads();
      for (int x = tid; x < n * nbk; x += nth) {
        const int i = x / nbk, y = x - i * nbk, l1 = y / (lb + 1), l2 = y - l1 * (lb + 1);
        fab[x] = pw[i * (la + lb + 2) + la - l1] * pw[i * (la + lb + 2) + la + 1 + lb - l2];
      }
      __syncthreads();
      const double* R = A.rbuf + A.rbase + (q0 + i0 - A.pp_base) * (int64_t)nR;
      // primitive pairs with a zero prefactor have no coupling block: the others of the chunk, four bits each
      unsigned list = 0;
      int nlive = 0;
      for (int i = 0; i < n; ++i)
        if (pw[i * (la + lb + 2)] != 0.0) list |= (unsigned)i << (4 * nlive++);
      if (nlive == 0) continue;
      const bool first = !live;
      live = true;
      if (single) {
        for (int e = tid; e < A.nrs; e += nth) {
          const int src = __ldg(A.rs_src + e);
          const double v = R[src & 0xffff];
          Rt[e] = v;
          atomicMax(En + (src >> 16), (__double2hiint(v) >> 20) & 0x7ff);
        }
      } else if (G == 1) {
        for (int e = tid; e < nrt; e += nth) {
          const int src = __ldg(A.rt_src + e), ri = src & 0xffff, blk = src >> 16;
          double s = first ? 0.0 : Rt[e];
#pragma unroll 4
          for (int j = 0; j < nlive; ++j) {
            const int i = (list >> (4 * j)) & 15;
            s = fma(fab[i * nbk + blk], R[(int64_t)i * nR + ri], s);
          }
          Rt[e] = s;
        }
      } else {
        const int g = tid / nrt, e = tid - g * nrt;
        if (g < G) {
          const int src = __ldg(A.rt_src + e), ri = src & 0xffff, blk = src >> 16;
          double s = first ? 0.0 : part[tid];
          for (int j = g; j < nlive; j += G) {
            const int i = (list >> (4 * j)) & 15;
            s = fma(fab[i * nbk + blk], R[(int64_t)i * nR + ri], s);
          }
          part[tid] = s;
        }
      }
    }
    __syncthreads();
    if (live) {
      for (int e = tid; !single && e < nrt; e += nth) {
        const int blk = __ldg(A.rt_src + e) >> 16;
        double s;
        if (G == 1) {
          s = Rt[e];
        } else {
          s = part[e];
          for (int g = 1; g < G; ++g) s += part[g * nrt + e];
          Rt[e] = s;
        }
        atomicMax(En + blk, (__double2hiint(s) >> 20) & 0x7ff);
      }
      __syncthreads();
      const int* srcs = single ? A.rs_src : A.rt_src;
      for (int e = tid; e < (single ? A.nrs : nrt); e += nth) {
        const int src = __ldg(srcs + e);
        const fx f = fx_of(Rt[e], En[src >> 16] + 2);
        Rx[e] = make_int2(f.h, f.l);
      }
      for (int e = tid; e < nbk; e += nth) {
        const int l1 = e / (lb + 1), mb = e - l1 * (lb + 1);
        int E = kNoScale;
        for (int l2 = mb; l2 <= lb; ++l2) {
          const double c = single ? tB[l2 * (lb + 1) + mb] * fab[l1 * (lb + 1) + l2] : tB[l2 * (lb + 1) + mb];
          const int ec = (__double2hiint(c) >> 20) & 0x7ff, n = En[scale_of(l1, l2)];
          if (ec == 0x7ff || n == 0x7ff)
            E = kNotFinite;
          else if (ec > 0 && n > 0)
            E = max(E, ec + n + 2 - 1023);
        }
        Ec[e] = E;
      }
      __syncthreads();
      for (int e = tid; e < nc; e += nth) {
        const int l1 = e / np, r = e - l1 * np;
        int l2 = 0;
        while ((l2 + 1) * (l2 + 2) / 2 <= r) ++l2;
        const int mb = r - l2 * (l2 + 1) / 2;
        const double c = single ? tB[l2 * (lb + 1) + mb] * fab[l1 * (lb + 1) + l2] : tB[l2 * (lb + 1) + mb];
        const fx f = fx_of(c, 1023 + Ec[l1 * (lb + 1) + mb] - En[scale_of(l1, l2)]);
        cx[e] = make_int2(f.h, f.l);
      }
      // coupling: rows r of one warp form one group: equal trip counts, one coalesced load per term
      int2 next = tid < nrp ? __ldg(A.rows + tid) : make_int2(0, 0);
      for (int r = tid; r < nrp; r += nth) {
        const int2 row = next;
        if (r + nth < nrp) next = __ldg(A.rows + r + nth);
        const int K = row.x >> 16;
        const int4* tp = A.terms + row.y;
        long long hh = 0, mid = 0;
#pragma unroll 4
        for (int j = 0; j < K; ++j) {
          const int4 g = __ldg(tp + 32 * j);
          const int2 v = Rx[single ? g.w : g.z];
          hh = fx_mad(g.x, v.x, hh);
          mid = fx_mad(g.x, v.y, mid);
          mid = fx_mad(g.y, v.x, mid);
        }
        if ((row.x & 0xffff) != 0xffff) {
          const fx f = fx_split(fx_sum(hh, mid));
          Wx[row.x & 0xffff] = make_int2(f.h, f.l);
        }
      }
      __syncthreads();
      for (int e = tid; e < na * na; e += nth) Dm[e] = rd[1 + rot_doff(la) + e];
      for (int e = tid; e < nDb; e += nth) Dm[na * na + e] = rd[1 + rot_doff(lb) + e];
      for (int e = tid; e < nWa * nb; e += nth) {
        const int q = (int)(((float)e + 0.5f) * inv_nwa), i1 = e - q * nWa, l1 = lo[i1];  // e / nWa (e < 2^12)
        const int amb = (q + 1) >> 1, mb = (q & 1) ? amb : -amb;
        const int E = Ec[l1 * (lb + 1) + amb];
        long long hh = 0, mid = 0;
        for (int l2 = amb; l2 <= lb; ++l2) {
          const int2 u = Wx[i1 * ws + l2 * l2 + l2 + mb], c = cx[l1 * np + l2 * (l2 + 1) / 2 + amb];
          hh = fx_mad(u.x, c.x, hh);
          mid = fx_mad(u.x, c.y, mid);
          mid = fx_mad(u.y, c.x, mid);
        }
        Zb[i1 * nb + mb + lb] = E == kNotFinite ? __longlong_as_double(0x7ff8000000000000ll)
                                : E == kNoScale ? 0.0
                                                : fx_double(fx_sum(hh, mid), E + 2 - 1023 - kFxBits);
      }
      __syncthreads();
    }
    if (!live) {
      // every primitive pair skipped: the block is zero (and omitted from a block-sparse output)
      if (A.mv.blk_off) return;
      const int64_t fa0 = A.shell_foff[a], fb0 = A.shell_foff[b];
      int64_t obase, ld;
      mol_output(A.mv, pr, obase, ld);
      double* o = A.out + obase;
      for (int e = tid; e < na * nb; e += nth) {
        const int ma = e / nb, mb = e % nb;
        o[(fa0 + ma) * ld + fb0 + mb] = 0.0;
        if (a != b) o[(fb0 + mb) * ld + fa0 + ma] = 0.0;
      }
      return;
    }
    // V' = t_A Z (diagonal in m); threads ordered by |m| so that the lanes of a warp run loops of nearly equal length
    for (int e = tid; e < na * nb; e += nth) {
      const int q = e / nb, mb = e - q * nb;
      const int ama = (q + 1) >> 1, ma = (q & 1) ? ama : -ama;
      double s = 0.0;
      for (int l1 = ama; l1 <= la; ++l1) s = fma(tA[l1 * (la + 1) + ama], Zb[(l1 * l1 + l1 + ma) * nb + mb], s);
      Vp[(ma + la) * nb + mb] = s;
    }
    __syncthreads();
    // back to the molecular frame: V = D^{la} V' (D^{lb})^T
    const double* Db = la != lb ? Dm + na * na : Dm;
    for (int e = tid; e < na * nb; e += nth) {
      const int ma = e / nb, mb = e % nb;
      double s = 0.0;
      for (int k = 0; k < nb; ++k) s = fma(Vp[ma * nb + k], Db[mb * nb + k], s);
      Yb[e] = s;
    }
    __syncthreads();
    for (int e = tid; e < na * nb; e += nth) {
      const int ma = e / nb, mb = e % nb;
      double s = 0.0;
      for (int k = 0; k < na; ++k) s = fma(Dm[ma * na + k], Yb[k * nb + mb], s);
      Vp[e] = s;
    }
    __syncthreads();
    if (A.mv.blk_off) {
      // block-sparse output: the block alone, row-major
      const int64_t off = A.mv.blk_off[pr];
      if (off < 0) return;
      double* o = A.out + off;
      for (int e = tid; e < na * nb; e += nth) {
        const int ma = e / nb, mb = e % nb;
        o[e] = (a == b && ma > mb) ? Vp[mb * nb + ma] : Vp[e];
      }
      return;
    }
    const int64_t fa0 = A.shell_foff[a], fb0 = A.shell_foff[b];
    int64_t obase, ld;
    mol_output(A.mv, pr, obase, ld);
    double* o = A.out + obase;
    for (int e = tid; e < na * nb; e += nth) {
      const int ma = e / nb, mb = e % nb;
      // diagonal shell block: the upper triangle serves both halves (exact symmetry)
      const double v = (a == b && ma > mb) ? Vp[mb * nb + ma] : Vp[e];
      o[(fa0 + ma) * ld + fb0 + mb] = v;
      if (a != b) o[(fb0 + mb) * ld + fa0 + ma] = v;
    }
  });
}

}  // namespace

int pair_threads(int la, int lb) {
  const int nW = (la + 1) * (la + 1) * (lb + 1) * (lb + 1);
  return nW >= 400 ? 128 : (nW >= 100 ? 64 : 32);
}

cudaError_t launch_pair_block(const PairArgs& args, int grid, cudaStream_t stream) {
  const int nth = pair_threads(args.la, args.lb);
  k_pair_block<<<grid, nth, pair_layout(args.la, args.lb, args.nrt, nth).bytes, stream>>>(args);
  return cudaGetLastError();
}

cudaError_t pair_block_setup() { return set_max_dynamic_smem((const void*)k_pair_block); }

}  // namespace shgo
