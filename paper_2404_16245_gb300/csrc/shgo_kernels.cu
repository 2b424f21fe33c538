// Once-per-basis kernels of the SHGO path (S1: Gaussian products, rotations of the pair frames), the launches of V and the
// four-centre electron-repulsion integrals (sm_103a, FP64).  The nucleus loop (S2) is in shgo_coupling.cu and
// shgo_coupling_f32.cu, the coupling, translation and write (S3 to S5) in shgo_pair.cu, the potential in shgo_esp.cu, the
// derivatives in shgo_deriv.cu, overlap and two-centre Coulomb integrals in shgo_twocentre.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <string>

#include "shgo_internal.h"
#include "shgo_math.h"

namespace shgo {

__constant__ HarmCoef c_harm;
__constant__ BoysConst c_boys;
__constant__ int c_lof[(kLmax + 1) * (kLmax + 1)];  // l of a packed harmonic index (l <= 8)

namespace {

constexpr double kTwoPi = 6.283185307179586476925286766559;


// |B - A|^2 and K_AB = exp(-alpha beta/(alpha + beta) |B - A|^2) of Eq. 5, with every operation
// rounded explicitly so that the coupling and pair kernels agree bit for bit on which primitive
// pairs have K_AB == 0 (the coupling kernel skips those, the pair kernel never reads them).
__device__ __forceinline__ double pair_ab2(const double* __restrict__ xyz, int a, int b) {
  const double dx = __dsub_rn(xyz[3 * b], xyz[3 * a]);
  const double dy = __dsub_rn(xyz[3 * b + 1], xyz[3 * a + 1]);
  const double dz = __dsub_rn(xyz[3 * b + 2], xyz[3 * a + 2]);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}
__device__ __forceinline__ double prim_kab(double ea, double eb, double ab2) {
  return exp(-__dmul_rn(__ddiv_rn(__dmul_rn(ea, eb), __dadd_rn(ea, eb)), ab2));
}

// Bound on every element of one primitive pair's block, per unit of total nuclear charge:
// |S_lm(r)| <= |r|^l (Racah normalisation) and |r_A| <= r_P + |PA|, and the potential of a non-negative
// radial density at any point is at most its value at the centre, int f(r)/r d^3r; so
//   |<a_i|1/|r-C||b_j>| <= |c_i c_j| K_AB 4 pi int_0^inf (r + |PA|)^la (r + |PB|)^lb e^{-p r^2} r dr.
// The overlap integrand is bounded the same way with r^2 dr; the larger of the two is returned.
// Moments: int_0^inf r^n e^{-p r^2} dr = M_n with M_0 = sqrt(pi/p)/2, M_1 = 1/(2p),
// M_{n+2} = (n+1)/(2p) M_n.
__device__ double prim_pair_bound(int la, int lb, double pa, double pb, double p, double pref) {
  double M[2 * kLmax + 4];
  M[0] = 0.5 * sqrt(3.14159265358979323846 / p);
  M[1] = 0.5 / p;
  for (int n = 0; n + 2 < 2 * kLmax + 4; ++n) M[n + 2] = (n + 1) * M[n] * (0.5 / p);
  double i1 = 0.0, i2 = 0.0, ca = 1.0;  // ca = C(la, i) pa^(la-i)
  double pa_pow[kLmax + 1], pb_pow[kLmax + 1];
  pa_pow[0] = pb_pow[0] = 1.0;
  for (int k = 1; k <= kLmax; ++k) {
    pa_pow[k] = pa_pow[k - 1] * pa;
    pb_pow[k] = pb_pow[k - 1] * pb;
  }
  for (int i = 0; i <= la; ++i) {
    ca = (i == 0) ? 1.0 : ca * (la - i + 1) / i;
    double cb = 1.0;
    for (int j = 0; j <= lb; ++j) {
      cb = (j == 0) ? 1.0 : cb * (lb - j + 1) / j;
      const double w = ca * cb * pa_pow[la - i] * pb_pow[lb - j];
      i1 += w * M[i + j + 1];
      i2 += w * M[i + j + 2];
    }
  }
  return fabs(pref) * 4.0 * 3.14159265358979323846 * fmax(i1, i2);
}

// Step S1, once per basis: the Gaussian-product data of every primitive pair.  A primitive pair whose
// bound (prim_pair_bound) is below kPrimSkip gets pref = 0, which every kernel treats as "skip": it
// changes any V element by at most kPrimSkip x sum |Z_C| (and any S element by at most kPrimSkip).
__global__ void k_pair_build(int64_t npp, const int* __restrict__ pp_pair, const int* __restrict__ pp_ij,
                             const int* __restrict__ pair_a, const int* __restrict__ pair_b,
                             const double* __restrict__ shell_xyz, const int* __restrict__ shell_l,
                             const int* __restrict__ shell_poff, const double* __restrict__ prim_exp,
                             const double* __restrict__ prim_coef, int use_bound, PPData* __restrict__ ppd) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < npp; q += (int64_t)gridDim.x * blockDim.x) {
    const int pr = pp_pair[q], ij = pp_ij[q];
    const int a = pair_a[pr], b = pair_b[pr];
    const int ia = shell_poff[a] + (ij >> 8), ib = shell_poff[b] + (ij & 255);
    const double ea = prim_exp[ia], eb = prim_exp[ib];
    const double ab2 = pair_ab2(shell_xyz, a, b);
    PPData d;
    d.p = ea + eb;
    d.rp = 1.0 / d.p;
    d.sp = sqrt(d.p);
    d.kab = prim_kab(ea, eb, ab2);
    d.pref = prim_coef[ia] * prim_coef[ib] * d.kab;
    d.ra = eb * d.rp;
    d.rb = ea * d.rp;
    const double ab = sqrt(ab2);
    d.shift = d.ra * ab;
    if (use_bound && d.pref != 0.0 &&
        prim_pair_bound(shell_l[a], shell_l[b], d.shift, d.rb * ab, d.p, d.pref) < kPrimSkip)
      d.pref = 0.0;
    ppd[q] = d;
  }
}

// Per shell pair: whether any of its primitive pairs is kept (the block-sparse layout's criterion, the same
// test the pair kernel applies before writing a block).
__global__ void k_pair_live(int64_t npairs, const int64_t* __restrict__ pair_ppoff, int64_t npp_total,
                            const PPData* __restrict__ ppd, uint8_t* __restrict__ live) {
  for (int64_t pr = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; pr < npairs;
       pr += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q1 = pr + 1 < npairs ? pair_ppoff[pr + 1] : npp_total;
    uint8_t any = 0;
    for (int64_t q = pair_ppoff[pr]; q < q1 && !any; ++q) any = ppd[q].pref != 0.0;
    live[pr] = any;
  }
}

// Per class (classes given by their first pair, pair_cls[c] .. pair_cls[c + 1]): live primitive pairs
// (pref != 0), shell pairs with at least one, and the sum over live primitive pairs of their
// molecule's nucleus count (batches; 0 otherwise).
__global__ void k_live_counts(int npairs, int ncls, const int* __restrict__ pair_cls,
                              const int64_t* __restrict__ pair_ppoff, int64_t npp_total,
                              const PPData* __restrict__ ppd, const int* __restrict__ pair_mol,
                              const int64_t* __restrict__ mol_nc, unsigned long long* __restrict__ live_pp,
                              unsigned long long* __restrict__ live_pairs, double* __restrict__ live_cent) {
  for (int pr = blockIdx.x * blockDim.x + threadIdx.x; pr < npairs; pr += gridDim.x * blockDim.x) {
    int c = 0;
    while (c + 1 < ncls && pair_cls[c + 1] <= pr) ++c;
    const int64_t q1 = pr + 1 < npairs ? pair_ppoff[pr + 1] : npp_total;
    unsigned long long n = 0;
    for (int64_t q = pair_ppoff[pr]; q < q1; ++q) n += ppd[q].pref != 0.0;
    if (n) {
      atomicAdd(live_pp + c, n);
      atomicAdd(live_pairs + c, 1ull);
      if (pair_mol) atomicAdd(live_cent + c, (double)n * (double)mol_nc[pair_mol[pr]]);
    }
  }
}

// Real rotation matrices D^l(R), l <= lm, R = Q^T (row-major in Rq), for the block's threads:
// D^0 = 1, D^1 from R, then D^{l+1} from D^l through the harmonic part of u_c S_{l,m'}(u) (the
// Gaunt product rule with one factor of degree 1).  Ends without a barrier after the last level.
__device__ void build_rotations(int lm, const double* Rq, double* Dm, const int* __restrict__ rot_ptr,
                                const GTerm* __restrict__ rot_terms) {
  const int tid = threadIdx.x, nth = blockDim.x;
  if (tid == 0) Dm[0] = 1.0;
  if (lm >= 1 && tid < 9) {
    const int m = tid / 3 - 1, c = tid % 3;  // row m, Cartesian column c (x, y, z)
    const int crow = m == -1 ? 1 : (m == 0 ? 2 : 0);
    const int mp = c == 0 ? 1 : (c == 1 ? -1 : 0);
    Dm[1 + (m + 1) * 3 + (mp + 1)] = Rq[crow * 3 + c];
  }
  for (int l = 1; l < lm; ++l) {
    __syncthreads();
    const double* Dl = Dm + rot_doff(l);
    double* Dn = Dm + rot_doff(l + 1);
    const int n1 = 2 * l + 3;
    for (int e = tid; e < n1 * n1; e += nth) {
      const int m = e / n1 - (l + 1), M = e % n1 - (l + 1);
      const int q = rot_index(l, M);
      double s = 0.0;
      if (m >= -l && m <= l) {
        for (int t = rot_ptr[q]; t < rot_ptr[q + 1]; ++t) {
          const GTerm g = rot_terms[t];
          s = fma(g.coef * Rq[6 + g.ridx], Dl[(m + l) * (2 * l + 1) + g.pad + l], s);
        }
        s *= c_harm.a[harm_index(l, m)];
      } else {
        const double* top = Dl + (2 * l) * (2 * l + 1);  // row m = l
        const double* bot = Dl;                          // row m = -l
        for (int t = rot_ptr[q]; t < rot_ptr[q + 1]; ++t) {
          const GTerm g = rot_terms[t];
          const double rx = Rq[g.ridx], ry = Rq[3 + g.ridx];
          const double v = (m > 0) ? (rx * top[g.pad + l] - ry * bot[g.pad + l])
                                   : (ry * top[g.pad + l] + rx * bot[g.pad + l]);
          s = fma(g.coef, v, s);
        }
        s *= c_harm.c[l];
      }
      Dn[e] = s;
    }
  }
}

// Once per basis: |B - A| and the rotation matrices D^0 .. D^lmax of the pair frame of every ordered
// pair of centres (one block each; they depend on the two positions only).
__global__ void __launch_bounds__(64) k_pair_rotations(int n_sites, int lmax, const int* __restrict__ site_rep,
                                                       const int* __restrict__ pair_a, const int* __restrict__ pair_b,
                                                       const double* __restrict__ site_rot,
                                                       const double* __restrict__ shell_xyz,
                                                       const int* __restrict__ rot_ptr,
                                                       const GTerm* __restrict__ rot_terms, double* __restrict__ rotd) {
  extern __shared__ double smem[];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int64_t per = rot_block(lmax);
  const int nD = rot_doff(lmax + 1);
  double* Dm = smem;
  double* Rq = Dm + nD;
  for (int i = blockIdx.x; i < n_sites; i += gridDim.x) {
    const int pr = site_rep[i];
    __syncthreads();
    if (tid < 9) Rq[tid] = site_rot[9 * i + (tid % 3) * 3 + tid / 3];
    __syncthreads();
    build_rotations(lmax, Rq, Dm, rot_ptr, rot_terms);
    __syncthreads();
    double* o = rotd + (int64_t)i * per;
    if (tid == 0) o[0] = sqrt(pair_ab2(shell_xyz, pair_a[pr], pair_b[pr]));
    for (int e = tid; e < nD; e += nth) o[1 + e] = Dm[e];
  }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Device tables
// ---------------------------------------------------------------------------------------------
namespace {
std::mutex g_tab_mu;
DeviceTables g_tabs[64];
bool g_tab_ok[64] = {};

template <typename T>
cudaError_t upload(T** dst, const std::vector<T>& src) {
  cudaError_t e = cudaMalloc((void**)dst, sizeof(T) * (src.empty() ? 1 : src.size()));
  if (e != cudaSuccess) return e;
  if (!src.empty()) e = cudaMemcpy(*dst, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice);
  return e;
}
}  // namespace

shgo_status device_tables(int device, const DeviceTables** out, std::string* err) {
  if (device < 0 || device >= 64) {
    *err = "device ordinal out of range";
    return SHGO_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lk(g_tab_mu);
  if (g_tab_ok[device]) {
    *out = &g_tabs[device];
    return SHGO_OK;
  }
  const Tables& t = tables_host();
  DeviceTables d;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = upload(&d.boys, t.boys);
  if (e == cudaSuccess) e = upload(&d.etab, t.etab);
  if (e == cudaSuccess) e = upload(&d.eoff, t.eoff);
  if (e == cudaSuccess) e = upload(&d.g_rowinfo, t.g_rowinfo);
  if (e == cudaSuccess) e = upload(&d.g_grp, t.g_grp);
  if (e == cudaSuccess) e = upload(&d.gt_ptr, t.gt_ptr);
  if (e == cudaSuccess) e = upload(&d.gt_terms, t.gt_terms);
  if (e == cudaSuccess) e = upload(&d.g_terms, t.g_terms);
  if (e == cudaSuccess) e = upload(&d.rmap, t.rmap);
  if (e == cudaSuccess) e = upload(&d.rnorm, t.rnorm);
  if (e == cudaSuccess) e = upload(&d.rot_ptr, t.rot_ptr);
  if (e == cudaSuccess) e = upload(&d.rot_terms, t.rot_terms);
  if (e == cudaSuccess) e = upload(&d.c2_ptr, t.c2_ptr);
  if (e == cudaSuccess) e = upload(&d.c2_terms, t.c2_terms);
  if (e == cudaSuccess) e = upload(&d.c2_a, t.c2_a);
  if (e == cudaSuccess) e = upload(&d.cx_rows, t.cx_rows);
  if (e == cudaSuccess) e = upload(&d.cx_terms, t.cx_terms);
  if (e == cudaSuccess) e = upload(&d.eri_eps, t.eri_eps);
  if (e == cudaSuccess) e = upload(&d.c2_cbase, t.c2_base);
  if (e == cudaSuccess) e = upload(&d.boys_ff, boys_table_pairs(t.boys));
  if (e == cudaSuccess) e = upload(&d.exp_ff, exp_table_pairs());
  if (e == cudaSuccess) e = upload(&d.rnorm_ff, pairs_of(t.rnorm));
  if (e == cudaSuccess) e = upload(&d.f32_items, coupling_f32_items(t.rmap_off));
  if (e == cudaSuccess) e = upload(&d.d_map0, t.d_map0);
  if (e == cudaSuccess) e = upload(&d.d_mapm, t.d_mapm);
  if (e == cudaSuccess) e = upload(&d.d_raise, t.d_raise);
  if (e == cudaSuccess) e = upload(&d.d_field, t.d_field);
  if (e == cudaSuccess) e = upload(&d.d_low, t.d_low);
  if (e == cudaSuccess) e = upload(&d.axial, t.axial);
  if (e == cudaSuccess) e = upload(&d.rt_src, t.rt_src);
  if (e == cudaSuccess) e = upload(&d.rs_src, t.rs_src);
  if (e == cudaSuccess) e = upload(&d.px_rows, t.px_rows);
  if (e == cudaSuccess) e = upload(&d.px_terms, t.px_terms);
  if (e == cudaSuccess) e = upload(&d.dt_ptr, t.dt_ptr);
  if (e == cudaSuccess) e = upload(&d.dt_terms, t.dt_terms);
  if (e == cudaSuccess) e = upload(&d.fr_terms, t.fr_terms);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_harm, &harm_coef_host(), sizeof(HarmCoef));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_boys, &boys_const_host(), sizeof(BoysConst));
  if (e == cudaSuccess) e = coupling_fp64_setup();
  if (e == cudaSuccess) e = esp_fp64_setup();
  if (e == cudaSuccess) e = twocentre_setup();
  if (e == cudaSuccess) e = pair_block_setup();
  if (e == cudaSuccess) e = coupling_f32_setup();
  if (e == cudaSuccess) {
    int lof[(kLmax + 1) * (kLmax + 1)];
    for (int l = 0; l <= kLmax; ++l)
      for (int m = -l; m <= l; ++m) lof[harm_index(l, m)] = l;
    e = cudaMemcpyToSymbol(c_lof, lof, sizeof(lof));
  }
  if (e != cudaSuccess) {
    *err = std::string("uploading tables: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? SHGO_ERR_OOM : SHGO_ERR_CUDA;
  }
  g_tabs[device] = d;
  g_tab_ok[device] = true;
  *out = &g_tabs[device];
  return SHGO_OK;
}

// The __constant__ recursion coefficients and Boys constants on the current device, without any
// allocation (used by the allocation-free entry point, which keeps its tables elsewhere).
shgo_status upload_constants(std::string* err) {
  cudaError_t e = cudaMemcpyToSymbol(c_harm, &harm_coef_host(), sizeof(HarmCoef));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_boys, &boys_const_host(), sizeof(BoysConst));
  if (e == cudaSuccess) e = coupling_fp64_setup();
  if (e == cudaSuccess) e = pair_block_setup();
  if (e == cudaSuccess) {
    int lof[(kLmax + 1) * (kLmax + 1)];
    for (int l = 0; l <= kLmax; ++l)
      for (int m = -l; m <= l; ++m) lof[harm_index(l, m)] = l;
    e = cudaMemcpyToSymbol(c_lof, lof, sizeof(lof));
  }
  if (e != cudaSuccess) {
    *err = std::string("uploading constants: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}

// ---------------------------------------------------------------------------------------------
// Launch
// ---------------------------------------------------------------------------------------------
static int grid_cap(int64_t n, int per_sm) {
  static int nsm = 0;
  if (nsm == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (nsm <= 0) nsm = 152;
  }
  const int64_t cap = (int64_t)nsm * per_sm;
  return (int)(n < cap ? n : cap);
}

namespace {
constexpr int kPoolStreams = 16;
std::mutex g_pool_mu;
cudaStream_t g_pool[64][kPoolStreams];
bool g_pool_ok[64] = {};

// Per-device pool of non-blocking streams on which the classes of one call run concurrently.
cudaError_t stream_pool(cudaStream_t** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (!g_pool_ok[dev]) {
    for (int i = 0; i < kPoolStreams; ++i) {
      e = cudaStreamCreateWithFlags(&g_pool[dev][i], cudaStreamNonBlocking);
      if (e != cudaSuccess) return e;
    }
    g_pool_ok[dev] = true;
  }
  *out = g_pool[dev];
  return cudaSuccess;
}

}  // namespace

cudaError_t pool_streams(cudaStream_t** out, int* n) {
  *n = kPoolStreams;
  return stream_pool(out);
}

int grid_cap_sm(int64_t n, int per_sm) { return grid_cap(n, per_sm); }

namespace {
struct Launcher {
  const DeviceBasis& db;
  const DeviceTables& dt;
  const Tables& th;
  MolView mv;
  const double* centers;
  const double* charges;
  double* out;


  // Work queue of class c's coupling (which = 0) or pair (which = 1) launch.  A launch over the whole
  // class of a batch takes its work from the queue in the batch's cost order; the uniform work of one
  // molecule, and the pieces of a class whose coupling buffer is split into regions, stride instead.
  // All keep the time limit.
  // Without a limit and without a queue the launch is the plain strided one (no atomics, no clock).
  WorkQueue queue(const ClassWork& w, size_t c, int which) const {
    WorkQueue q;
    const int* items = which == 0 ? db.cp_items : db.pr_items;
    const bool timed = db.limit_ns != ~0ull, queued = db.region == 0 && items;
    if (!db.ctrl || (!timed && !queued)) return q;
    unsigned char* slot = db.ctrl + kCtrlHead + kCtrlSlot * (2 * c + (size_t)which);
    if (timed) {
      q.t0 = reinterpret_cast<unsigned long long*>(slot + 8);
      q.err = reinterpret_cast<int*>(db.ctrl);
      q.limit_ns = db.limit_ns;
    }
    if (queued) {
      q.qctr = reinterpret_cast<unsigned long long*>(slot);
      q.items = items + (which == 0 ? w.pp_base : (int64_t)w.pair_base);
    }
    return q;
  }
  // Clears class c's two queue slots on `s` (before launching the class again within one call).
  cudaError_t reset(size_t c, cudaStream_t s) const {
    if (!db.ctrl || (db.limit_ns == ~0ull && !db.cp_items && !db.pr_items)) return cudaSuccess;
    return cudaMemsetAsync(db.ctrl + kCtrlHead + kCtrlSlot * 2 * c, 0, 2 * kCtrlSlot, s);
  }

  void coupling(const ClassWork& w, size_t c, int64_t rbase, cudaStream_t s) const {
    if (w.npp == 0) return;
    const int lam = w.la + w.lb;
    const int* rmap = dt.rmap + th.rmap_off[lam];
    CouplingArgs a;
    a.q = queue(w, c, 0);
    a.npp = w.npp;
    a.pp_base = w.pp_base;
    a.rbase = rbase;
    a.pp_pair = db.pp_pair;
    a.pair_a = db.pair_a;
    a.shell_xyz = db.shell_xyz;
    a.mv = mv;
    a.centers = centers;
    a.charges = charges;
    a.rmap = rmap;
    a.rnorm = dt.rnorm + th.rmap_off[lam];
    a.site_rot = db.site_rot;
    a.pair_site = db.pair_site;
    a.ppd = db.ppd;
    a.rbuf = db.rbuf;
    a.small_blocks_ok = db.f32_small_blocks;
    if (db.precision != SHGO_PREC_FP64) {
      a.boys_ff = dt.boys_ff;
      a.exp_ff = dt.exp_ff;
      a.items = dt.f32_items + th.rmap_off[lam];
      a.rnorm_ff = dt.rnorm_ff + th.rmap_off[lam];
      launch_coupling_f32(lam, db.precision == SHGO_PREC_FP32_BULK, a, grid_cap(w.npp, 8), s);
      return;
    }
    launch_coupling_fp64(lam, a, s);
  }
  void pair(const ClassWork& w, size_t c, int64_t rbase, cudaStream_t s) const {
    if (w.npairs == 0) return;
    const int cid = class_id(w.la, w.lb);
    PairArgs p;
    p.la = w.la;
    p.lb = w.lb;
    p.npairs = w.npairs;
    p.pair_base = w.pair_base;
    p.pp_base = w.pp_base;
    p.rbase = rbase;
    p.rot_per = rot_block(db.rot_lmax);
    p.pair_a = db.pair_a;
    p.pair_b = db.pair_b;
    p.pair_ppoff = db.pair_ppoff;
    p.pair_site = db.pair_site;
    p.rotd = db.rotd;
    p.shell_nprim = db.shell_nprim;
    p.shell_foff = db.shell_foff;
    p.axial = dt.axial;
    p.nrt = th.rt_base[cid + 1] - th.rt_base[cid];
    p.rt_src = dt.rt_src + th.rt_base[cid];
    p.nrs = th.rs_base[cid + 1] - th.rs_base[cid];
    p.rs_src = dt.rs_src + th.rs_base[cid];
    p.rows = dt.px_rows + th.g_rowbase[cid];
    p.terms = dt.px_terms + th.g_termbase[cid];
    p.ppd = db.ppd;
    p.rbuf = db.rbuf;
    p.mv = mv;
    p.out = out;
    p.wq = queue(w, c, 1);
    launch_pair_block(p, grid_cap(w.npairs, 16), s);
  }
};

// Clears the queue slots of a basis's control block (counters, start times) on `stream`; the error word
// stays set until the host reads it.
cudaError_t clear_ctrl(const DeviceBasis& db, size_t nclasses, cudaStream_t stream) {
  if (!db.ctrl || (db.limit_ns == ~0ull && !db.cp_items && !db.pr_items)) return cudaSuccess;
  return cudaMemsetAsync(db.ctrl + kCtrlHead, 0, ctrl_bytes(nclasses) - kCtrlHead, stream);
}

// Pieces of a class whose coupling blocks fit `region` doubles, cut between shell pairs.
std::vector<ClassWork> class_chunks(const ClassWork& w, const int64_t* ppoff, int64_t region) {
  std::vector<ClassWork> out;
  const int64_t nR = n_r(w.la + w.lb);
  int q = w.pair_base;
  const int qend = w.pair_base + w.npairs;
  while (q < qend) {
    ClassWork ch{w.la, w.lb, 0, q, 0, ppoff[q]};
    int64_t used = 0;
    while (q < qend && (ch.npairs == 0 || used + (ppoff[q + 1] - ppoff[q]) * nR <= region)) {
      used += (ppoff[q + 1] - ppoff[q]) * nR;
      ++ch.npairs;
      ++q;
    }
    ch.npp = ppoff[q] - ch.pp_base;
    out.push_back(ch);
  }
  return out;
}

// Fork the work of `order` over the pool streams after the work already queued on `stream`, and
// make `stream` wait for all of it.  phase: 0 = coupling only, 1 = pair blocks only, 2 = both.
// With a bounded coupling buffer (db.region > 0) stream i uses region i and runs each of its
// classes chunk by chunk (both kernels per chunk; phase must be 2).
cudaError_t run_concurrent(const Launcher& L, const std::vector<ClassWork>& work, const std::vector<int64_t>& rbases,
                           const std::vector<int>& order, int phase, cudaStream_t stream) {
  cudaStream_t* pool = nullptr;
  cudaError_t e = stream_pool(&pool);
  if (e != cudaSuccess) return e;
  const int ns = (int)std::min<size_t>(order.size(), (size_t)kPoolStreams);
  if (ns == 0) return cudaSuccess;
  cudaEvent_t fork;
  e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  if (e != cudaSuccess) return e;
  cudaEventRecord(fork, stream);
  for (int i = 0; i < ns; ++i) cudaStreamWaitEvent(pool[i], fork, 0);
  for (size_t k = 0; k < order.size(); ++k) {
    const int c = order[k];
    cudaStream_t s = pool[k % ns];
    if (L.db.region > 0) {
      const int64_t rb = (int64_t)(k % ns) * L.db.region;
      for (const ClassWork& ch : class_chunks(work[c], L.db.h_ppoff, L.db.region)) {
        L.coupling(ch, c, rb, s);
        L.pair(ch, c, rb, s);
      }
      continue;
    }
    if (phase != 1) L.coupling(work[c], c, rbases[c], s);
    if (phase != 0) L.pair(work[c], c, rbases[c], s);
  }
  for (int i = 0; i < ns; ++i) {
    cudaEvent_t join;
    e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
    if (e != cudaSuccess) break;
    cudaEventRecord(join, pool[i]);
    cudaStreamWaitEvent(stream, join, 0);
    cudaEventDestroy(join);
  }
  cudaEventDestroy(fork);
  return e;
}

std::vector<int64_t> class_rbases(const std::vector<ClassWork>& work) {
  std::vector<int64_t> rbases(work.size());
  int64_t rbase = 0;
  for (size_t c = 0; c < work.size(); ++c) {
    rbases[c] = rbase;
    rbase += work[c].npp * n_r(work[c].la + work[c].lb);
  }
  return rbases;
}

// Classes by decreasing estimated cost (dealt round-robin over the pool streams).
std::vector<int> class_order(const std::vector<ClassWork>& work, double nuclei_per_pair) {
  std::vector<int> order(work.size());
  std::vector<double> cost(work.size());
  for (size_t c = 0; c < work.size(); ++c) {
    order[c] = (int)c;
    const int lam = work[c].la + work[c].lb;
    const double nW = (double)(work[c].la + 1) * (work[c].la + 1) * (work[c].lb + 1) * (work[c].lb + 1);
    cost[c] = (double)work[c].npp * (nuclei_per_pair * n_r(lam) + 8.0 * nW) + (double)work[c].npairs * 30.0 * nW;
  }
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
  return order;
}

shgo_status launch_error(std::string* err) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    *err = std::string("kernel launch: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}
}  // namespace

shgo_status launch_nuclear_attraction(const DeviceBasis& db, const DeviceTables& dt,
                                      const std::vector<ClassWork>& work, int64_t nbf, int64_t ncenters,
                                      const double* centers, const double* charges, double* out,
                                      cudaStream_t stream, std::string* err, cudaEvent_t* events, bool concurrent,
                                      const int64_t* blk_off, int64_t out_doubles) {
  if (events) cudaEventRecord(events[0], stream);
  if (nbf == 0 || ncenters == 0) {
    if (events) cudaEventRecord(events[1], stream);
  }
  if (nbf == 0) {
    if (events) cudaEventRecord(events[2], stream);
    return SHGO_OK;
  }
  if (ncenters == 0) {
    const size_t n = blk_off ? (size_t)out_doubles : (size_t)nbf * (size_t)nbf;
    cudaError_t e = n ? cudaMemsetAsync(out, 0, sizeof(double) * n, stream) : cudaSuccess;
    if (events) cudaEventRecord(events[2], stream);
    if (e != cudaSuccess) {
      *err = cudaGetErrorString(e);
      return SHGO_ERR_CUDA;
    }
    return SHGO_OK;
  }
  const Tables& th = tables_host();
  const std::vector<int64_t> rbases = class_rbases(work);
  MolView mv;
  mv.ncenters = ncenters;
  mv.nbf = nbf;
  mv.blk_off = blk_off;
  const Launcher L{db, dt, th, mv, centers, charges, out};
  cudaError_t e = clear_ctrl(db, work.size(), stream);
  if (events && db.region > 0) {
    *err = "phase timing needs the whole coupling buffer; this basis uses bounded regions";
    return SHGO_ERR_INVALID_ARG;
  }
  if (e != cudaSuccess) {
  } else if (!concurrent) {
    for (size_t c = 0; c < work.size(); ++c) L.coupling(work[c], c, rbases[c], stream);
    if (events) cudaEventRecord(events[1], stream);
    for (size_t c = 0; c < work.size(); ++c) L.pair(work[c], c, rbases[c], stream);
  } else {
    const std::vector<int> order = class_order(work, (double)ncenters);
    if (events) {
      e = run_concurrent(L, work, rbases, order, 0, stream);
      cudaEventRecord(events[1], stream);
      if (e == cudaSuccess) e = run_concurrent(L, work, rbases, order, 1, stream);
    } else {
      e = run_concurrent(L, work, rbases, order, 2, stream);
    }
  }
  if (events) cudaEventRecord(events[2], stream);
  if (e != cudaSuccess) {
    *err = std::string("kernel launch: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return launch_error(err);
}

shgo_status launch_class_timed(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work,
                               const MolView& mv, const double* centers, const double* charges, double* out,
                               cudaStream_t stream, double* ms, std::string* err) {
  if (work.empty()) return SHGO_OK;
  const Tables& th = tables_host();
  const std::vector<int64_t> rbases = class_rbases(work);
  const Launcher L{db, dt, th, mv, centers, charges, out};
  std::vector<cudaEvent_t> ev(3 * work.size(), nullptr);
  cudaError_t e = clear_ctrl(db, work.size(), stream);
  for (auto& x : ev)
    if (e == cudaSuccess) e = cudaEventCreate(&x);
  for (size_t c = 0; c < work.size() && e == cudaSuccess; ++c) {
    cudaEventRecord(ev[3 * c], stream);
    L.coupling(work[c], c, rbases[c], stream);
    cudaEventRecord(ev[3 * c + 1], stream);
    L.pair(work[c], c, rbases[c], stream);
    cudaEventRecord(ev[3 * c + 2], stream);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaEventSynchronize(ev.back());
  for (size_t c = 0; c < work.size() && e == cudaSuccess; ++c) {
    float a = 0, b = 0;
    e = cudaEventElapsedTime(&a, ev[3 * c], ev[3 * c + 1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&b, ev[3 * c + 1], ev[3 * c + 2]);
    ms[2 * c] = a;
    ms[2 * c + 1] = b;
  }
  for (auto& x : ev)
    if (x) cudaEventDestroy(x);
  if (e != cudaSuccess) {
    *err = std::string("class timing: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return SHGO_OK;
}

shgo_status launch_batched(const DeviceBasis& db, const DeviceTables& dt, const std::vector<ClassWork>& work,
                           const MolView& mv, double nuclei_per_pair, const double* centers, const double* charges,
                           double* out, cudaStream_t stream, std::string* err) {
  if (work.empty()) return SHGO_OK;
  const Tables& th = tables_host();
  const std::vector<int64_t> rbases = class_rbases(work);
  const Launcher L{db, dt, th, mv, centers, charges, out};
  cudaError_t e = clear_ctrl(db, work.size(), stream);
  if (e == cudaSuccess) e = run_concurrent(L, work, rbases, class_order(work, nuclei_per_pair), 2, stream);
  if (e != cudaSuccess) {
    *err = std::string("kernel launch: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  return launch_error(err);
}

shgo_status launch_pair_rotations(const DeviceBasis& db, const DeviceTables& dt, cudaStream_t stream, std::string* err) {
  if (db.n_sites == 0) return SHGO_OK;
  const size_t sm = sizeof(double) * ((size_t)rot_doff(db.rot_lmax + 1) + 16);
  k_pair_rotations<<<grid_cap(db.n_sites, 16), 64, sm, stream>>>(db.n_sites, db.rot_lmax, db.site_rep, db.pair_a,
                                                                   db.pair_b, db.site_rot, db.shell_xyz, dt.rot_ptr,
                                                                   dt.rot_terms, db.rotd);
  return launch_error(err);
}

shgo_status launch_pair_build(const DeviceBasis& db, int64_t npp, cudaStream_t stream, std::string* err) {
  if (npp == 0) return SHGO_OK;
  const int64_t blocks = std::min<int64_t>((npp + 255) / 256, 152 * 32);
  k_pair_build<<<(int)blocks, 256, 0, stream>>>(npp, db.pp_pair, db.pp_ij, db.pair_a, db.pair_b, db.shell_xyz,
                                                 db.shell_l, db.shell_poff, db.prim_exp, db.prim_coef, db.prim_bound,
                                                 db.ppd);
  return launch_error(err);
}

shgo_status launch_pair_live(const DeviceBasis& db, int64_t npairs, int64_t npp, uint8_t* live, cudaStream_t stream,
                             std::string* err) {
  if (npairs == 0) return SHGO_OK;
  const int64_t blocks = std::min<int64_t>((npairs + 255) / 256, 152 * 32);
  k_pair_live<<<(int)blocks, 256, 0, stream>>>(npairs, db.pair_ppoff, npp, db.ppd, live);
  return launch_error(err);
}

shgo_status live_counts(const DeviceBasis& db, const std::vector<ClassWork>& work, int64_t npairs, int64_t npp,
                        const int* pair_mol, const int64_t* mol_nc, std::vector<int64_t>& live_pp,
                        std::vector<int64_t>& live_pairs, std::vector<double>& live_cent, std::string* err) {
  const int nc = (int)work.size();
  live_pp.assign(nc, 0);
  live_pairs.assign(nc, 0);
  live_cent.assign(nc, 0.0);
  if (nc == 0 || npairs == 0) return SHGO_OK;
  std::vector<int> cls(nc);
  for (int c = 0; c < nc; ++c) cls[c] = work[c].pair_base;
  // one scratch block: class starts, then the three counters
  const size_t b_cls = sizeof(int) * nc, b_cnt = sizeof(unsigned long long) * nc, b_cent = sizeof(double) * nc;
  unsigned char* scratch = nullptr;
  cudaError_t e = cudaMalloc((void**)&scratch, b_cls + 2 * b_cnt + b_cent + 64);
  if (e == cudaSuccess) e = cudaMemset(scratch, 0, b_cls + 2 * b_cnt + b_cent + 64);
  int* d_cls = reinterpret_cast<int*>(scratch);
  unsigned long long* d_pp = reinterpret_cast<unsigned long long*>(scratch + ((b_cls + 15) & ~(size_t)15));
  unsigned long long* d_pairs = d_pp + nc;
  double* d_cent = reinterpret_cast<double*>(d_pairs + nc);
  if (e == cudaSuccess) e = cudaMemcpy(d_cls, cls.data(), b_cls, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    const int64_t blocks = std::min<int64_t>((npairs + 255) / 256, 152 * 16);
    k_live_counts<<<(int)blocks, 256>>>((int)npairs, nc, d_cls, db.pair_ppoff, npp, db.ppd, pair_mol, mol_nc, d_pp,
                                        d_pairs, d_cent);
    e = cudaGetLastError();
  }
  std::vector<unsigned long long> hp(nc), hq(nc);
  if (e == cudaSuccess) e = cudaMemcpy(hp.data(), d_pp, b_cnt, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(hq.data(), d_pairs, b_cnt, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(live_cent.data(), d_cent, b_cent, cudaMemcpyDeviceToHost);
  cudaFree(scratch);
  if (e != cudaSuccess) {
    *err = std::string("counting live primitive pairs: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  for (int c = 0; c < nc; ++c) {
    live_pp[c] = (int64_t)hp[c];
    live_pairs[c] = (int64_t)hq[c];
  }
  return SHGO_OK;
}

// Real solid harmonics S_lm(x, y, z), l <= lmax, by columns: thread t of nth takes the columns
// m = t - lmax, t + nth - lmax, ...; each walks the diagonal chain S_{l+1,+-(l+1)} = c_l (x S_ll -+ y S_{l,-l})
// (S_11 = x, S_1-1 = y) up to |m| and then S_{l+1,m} = a_lm z S_lm - b_lm r^2 S_{l-1,m} (the recursion of
// solid_harmonics, whose entries it reproduces operation for operation) into S[l^2 + l + m].
__device__ void solid_harmonics_columns(int lmax, double x, double y, double z, double* S, int tid, int nth) {
  const double r2 = x * x + y * y + z * z;
  for (int col = tid; col < 2 * lmax + 1; col += nth) {
    const int m = col - lmax, am = m < 0 ? -m : m;
    double sp = 1.0, sm = 0.0;  // S_{l,l}, S_{l,-l}
    if (am >= 1) {
      sp = x;
      sm = y;
      for (int l = 1; l < am; ++l) {
        const double c = c_harm.c[l];
        const double np = c * (x * sp - y * sm), nm = c * (y * sp + x * sm);
        sp = np;
        sm = nm;
      }
    }
    double prv = 0.0, cur = m < 0 ? sm : sp;
    S[am * am + am + m] = cur;
    for (int l = am; l < lmax; ++l) {
      const int k = l * l + l + m;
      double v = c_harm.a[k] * (z * cur);
      if (m > -l && m < l) v -= c_harm.b[k] * (r2 * prv);
      S[(l + 1) * (l + 1) + l + 1 + m] = v;
      prv = cur;
      cur = v;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Four-centre electron-repulsion integrals (ab|cd) (Eqs. 13-15), in the SHGO form re-derived from
// Eqs. 3 and 7-8 (the printed Eq. 15 carries the same-centre coupling defect of Eq. 12):
//  1. Each pair is translated to its product centre (Eq. 7, real addition theorem) and its two
//     harmonics at P coupled by the Gaunt coefficients:
//       phi_a phi_b = c c' K_AB sum_{L,M,k} Y[L,M,k] r_P^{2k} S_LM(r_P) e^{-p r_P^2}.
//  2. r^{2k} S_LM e^{-pr^2} = sum_n eps_{k,n}(L) p^{-(k+n)} Laplacian^n [S_LM e^{-pr^2}], and by Eq. 3
//     S_LM(r_P) e^{-p r_P^2} = (2p)^{-L} S_LM(grad_P) e^{-p r_P^2}, so the pair is
//       sum_{L,M,n} D[L,M,n] Laplacian_P^n S_LM(grad_P) e^{-p r_P^2}
//     (k_eri_dist writes D per primitive pair and block entry (ma, mb)).
//  3. For two such terms at P and Q, with R = P - Q and u = |R|^2, every operator acts on the s-s integral
//     g(u) = 2 pi^{5/2} / (p q sqrt(p + q)) F_0(rho u), rho = pq/(p + q), as grad_P = grad_R, grad_Q = -grad_R:
//       (-1)^{L2} Laplacian^{n1+n2} S_L1M1(grad) S_L2M2(grad) g
//         = (-1)^{L2} sum_{L,M} G(L1M1, L2M2; LM) 2^L S_LM(R) sum_j a_{K,j}(L) u^j g^{(L+K+j)}(u),
//     K = (L1 + L2 - L)/2 + n1 + n2 (product rule, Hobson's theorem and Laplacian_L of the two-centre
//     kernel), g^{(N)}(u) = 2 pi^{5/2} / (p q sqrt(p + q)) (-rho)^N F_N(rho u).
//  4. (ab|cd) = sum over primitive quartets of D_ab I D_cd^T (k_eri_part, summed by k_eri_reduce).
// The entries (L, M, n) of a pair use the (L, M, k) layout of the coupling buffer for Lambda = la + lb.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int lmk_first(int lam, int L) {
  int off = 0;
  for (int Lp = 0; Lp < L; ++Lp) off += (2 * Lp + 1) * (kmax_of(lam, Lp) + 1);
  return off;
}

__device__ __forceinline__ int l_of_index(int h) {
  int L = (int)sqrtf((float)h);
  while (L * L > h) --L;
  while ((L + 1) * (L + 1) <= h) ++L;
  return L;
}

// One primitive pair per block iteration: D[(ma mb) nr + e], e over the (L, M, n) entries of
// Lambda = la + lb, for the class's primitive pairs pp_base .. pp_base + npp (dist: the class block).
__global__ void __launch_bounds__(128) k_eri_dist(int la, int lb, int64_t npp, int64_t pp_base,
                                                  const int* __restrict__ pp_pair, const int* __restrict__ pp_ij,
                                                  const int* __restrict__ pair_a, const int* __restrict__ pair_b,
                                                  const double* __restrict__ shell_xyz,
                                                  const int* __restrict__ shell_poff,
                                                  const double* __restrict__ prim_exp,
                                                  const double* __restrict__ prim_coef, const double* __restrict__ etab,
                                                  const int* __restrict__ eoff, const int* __restrict__ gt_ptr,
                                                  const GTerm* __restrict__ gt_terms, const double* __restrict__ eps,
                                                  double* __restrict__ dist) {
  extern __shared__ double smem[];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lam = la + lb, na = 2 * la + 1, nb = 2 * lb + 1, nr = n_r(lam), nh = n_harm(lam);
  const int nha = n_harm(la), nhb = n_harm(lb), ws = w_stride(lb);
  double* S = smem;             // [nha] S_lm(B - A)
  double* EA = S + nha;         // [na][nha] translation of a to P
  double* EB = EA + na * nha;   // [nb][nhb] translation of b to P
  for (int64_t w = blockIdx.x; w < npp; w += gridDim.x) {
    const int64_t pp = pp_base + w;
    const int pr = pp_pair[pp], ij = pp_ij[pp];
    const int a = pair_a[pr], b = pair_b[pr];
    const int ia = shell_poff[a] + (ij >> 8), ib = shell_poff[b] + (ij & 255);
    const double al = prim_exp[ia], be = prim_exp[ib], p = al + be, ip = 1.0 / p;
    const double dx = shell_xyz[3 * b] - shell_xyz[3 * a], dy = shell_xyz[3 * b + 1] - shell_xyz[3 * a + 1],
                 dz = shell_xyz[3 * b + 2] - shell_xyz[3 * a + 2];
    __syncthreads();  // the previous primitive pair is done with S, EA, EB
    solid_harmonics_columns(la, dx, dy, dz, S, tid, nth);
    __syncthreads();
    // S_la,ma(r - A) = sum_{l1 m1} EA[ma][l1 m1] S_l1m1(r - P): P - A = (beta/p)(B - A)
    for (int e = tid; e < na * nha; e += nth) {
      const int ma = e / nha - la, i1 = e - (ma + la) * nha, l1 = c_lof[i1], m1 = i1 - l1 * l1 - l1, lr = la - l1;
      const double* t = etab + eoff[la] + translation_offset_dev(la, ma, l1, m1);
      double v = 0.0, f = 1.0;
      for (int nu = -lr; nu <= lr; ++nu) v = fma(t[nu + lr], S[lr * lr + lr + nu], v);
      for (int k = 0; k < lr; ++k) f *= be * ip;
      EA[e] = v * f;
    }
    // P - B = (alpha/p)(A - B) and S_l(A - B) = (-1)^l S_l(B - A)
    for (int e = tid; e < nb * nhb; e += nth) {
      const int mb = e / nhb - lb, i2 = e - (mb + lb) * nhb, l2 = c_lof[i2], m2 = i2 - l2 * l2 - l2, lr = lb - l2;
      const double* t = etab + eoff[lb] + translation_offset_dev(lb, mb, l2, m2);
      double v = 0.0, f = 1.0;
      for (int nu = -lr; nu <= lr; ++nu) v = fma(t[nu + lr], S[lr * lr + lr + nu], v);
      for (int k = 0; k < lr; ++k) f *= -al * ip;
      EB[e] = v * f;
    }
    __syncthreads();
    const double ab2 = dx * dx + dy * dy + dz * dz;
    const double pref = prim_coef[ia] * prim_coef[ib] * exp(-al * be * ip * ab2);
    double* out = dist + w * (int64_t)(na * nb) * nr;
    // one (ma mb, L, M) per thread: Y[L,M,k] for every k by the Gaunt coupling, then the Laplacian form
    for (int g = tid; g < na * nb * nh; g += nth) {
      const int mamb = g / nh, h = g - mamb * nh, L = c_lof[h], M = h - L * L - L, km = kmax_of(lam, L);
      const int ma = mamb / nb, mb = mamb - ma * nb;
      const int e0 = lmk_first(lam, L) + (M + L) * (km + 1);
      double Y[kC2K + 1];
#pragma unroll
      for (int k = 0; k <= kC2K; ++k) {
        double y = 0.0;
        if (k <= km)
          for (int t = gt_ptr[e0 + k]; t < gt_ptr[e0 + k + 1]; ++t) {
            const GTerm gtm = gt_terms[t];
            const int i1 = gtm.ridx / ws, i2 = gtm.ridx - i1 * ws;
            y = fma(gtm.coef * EA[ma * nha + i1], EB[mb * nhb + i2], y);
          }
        Y[k] = y;
      }
      double scale = pref;
      for (int k = 0; k < L; ++k) scale *= 0.5 * ip;
#pragma unroll
      for (int n = 0; n <= kC2K; ++n) {
        if (n > km) break;
        const double* en = eps + (size_t)L * (kC2K + 1) * (kC2K + 1) + n;
        double v = 0.0, pw = 1.0;
        for (int k = 0; k < 2 * n; ++k) pw *= ip;  // p^{-(k+n)} at k = n
#pragma unroll
        for (int k = 0; k <= kC2K; ++k) {
          if (k < n || k > km) continue;
          v = fma(en[k * (kC2K + 1)] * pw, Y[k], v);
          pw *= ip;
        }
        out[mamb * nr + e0 + n] = scale * v;
      }
    }
  }
}

size_t eri_dist_smem(int la, int lb) {
  return sizeof(double) * ((size_t)n_harm(la) + (2 * la + 1) * n_harm(la) + (2 * lb + 1) * n_harm(lb) + 8);
}

// Work item of k_eri_part: one bra primitive pair pp1 (of the bra class, in [pp_lo, pp_hi)), one slice of
// its bra entries (nslice slices of equal height) and one ket shell pair q2 (of the ket class, in
// [q2_lo, q2_hi)); for the same class only q2 <= q1 is needed.  The item computes the slice's rows of
// X = sum over the ket primitive pairs of I D_cd^T (I: the interaction matrix of step 3, built in tiles of
// kEriPartTile columns over (ket primitive pair, ket entry)) and writes its share of the block,
// D_ab[:, slice] X[slice, :], to part[(((pp1 - pp_lo) nslice + slice) n2w + q2 - q2_lo) nab ncd].
// Ket primitive pairs are taken `chunk` at a time: one thread per primitive pair for P - Q, its Boys values
// and the tables g^{(N)}(u), u^j; one thread per (primitive pair, column m) for the solid harmonics
// S_LM(P - Q); then the radial factors Z of all of them; then the tiles, contracted into X with 2 x 2
// register tiles (rows r, r + nxr and columns c, c + nxc).
constexpr int kEriPartTile = 32;
constexpr int kEriTileStride = kEriPartTile + 1;  // odd row stride: rows read together fall in distinct banks
constexpr size_t kEriSmemTarget = 56 * 1024;  // shared memory of a k_eri_part block (four per SM)

__global__ void __launch_bounds__(256) k_eri_part(
    int la, int lb, int lc, int ld, int64_t pp_lo, int64_t pp_hi, int base1, int q2_lo, int q2_hi, int same,
    int chunk, int nslice, const int* __restrict__ pp_pair, const int* __restrict__ pp_ij, const int* __restrict__ pair_a,
    const int* __restrict__ pair_b, const int64_t* __restrict__ pair_ppoff, int64_t pp_base1, int64_t pp_base2,
    int base2, const double* __restrict__ shell_xyz, const int* __restrict__ shell_poff,
    const int* __restrict__ shell_nprim, const double* __restrict__ prim_exp, const double* __restrict__ dist1,
    const double* __restrict__ dist2, const double* __restrict__ boys_tab, const int* __restrict__ rmap1,
    const int* __restrict__ rmap2, const int* __restrict__ rmapt, const int* __restrict__ c2_ptr,
    const int* __restrict__ c2_cbase, const GTerm* __restrict__ c2_terms, const double* __restrict__ c2_a,
    double* __restrict__ part) {
  extern __shared__ double smem[];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lam1 = la + lb, lam2 = lc + ld, lt = lam1 + lam2;
  const int nr1f = n_r(lam1), nr2 = n_r(lam2), nrt = n_r(lt), nht = n_harm(lt);
  const int nab = (2 * la + 1) * (2 * lb + 1), ncd = (2 * lc + 1) * (2 * ld + 1);
  const int n2w = q2_hi - q2_lo, rows = (nr1f + nslice - 1) / nslice;
  double* X = smem;                            // [rows][ncd]
  double* It = X + (size_t)rows * ncd;         // [rows][kEriTileStride]
  double* Dt = It + rows * kEriTileStride;     // [ncd][kEriTileStride] ket distributions of the tile
  double* S = Dt + ncd * kEriTileStride;       // [chunk][nht]
  double* F = S + (size_t)chunk * nht;         // [chunk][lt + 1]
  double* Z = F + (size_t)chunk * (lt + 1);    // [chunk][nrt]
  double* G = Z + (size_t)chunk * nrt;         // [chunk][lt + 1]: g^{(N)}(u) = cpq (-rho)^N F_N(rho u)
  double* U = G + (size_t)chunk * (lt + 1);    // [chunk][lt / 2 + 1]: u^j
  double* Rv = U + (size_t)chunk * (lt / 2 + 1);  // [chunk][3]: P - Q
  int* kap1 = (int*)(Rv + 3 * (size_t)chunk);    // bra entries: h | n << 12 | L << 20
  int* kap2 = kap1 + nr1f;                     // ket entries
  int* zoff = kap2 + nr2;                      // [lt + 1]
  for (int e = tid; e < nr1f; e += nth) {
    const int r = rmap1[e], h = r & 0xfff;
    kap1[e] = h | ((r >> 24) << 12) | (l_of_index(h) << 20);
  }
  for (int e = tid; e < nr2; e += nth) {
    const int r = rmap2[e], h = r & 0xfff;
    kap2[e] = h | ((r >> 24) << 12) | (l_of_index(h) << 20);
  }
  if (tid <= lt) zoff[tid] = lmk_first(lt, tid);
  const int64_t nitems = (pp_hi - pp_lo) * nslice * n2w;
  for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int64_t row = it / n2w, pp1 = pp_lo + row / nslice;
    const int slice = (int)(row - (row / nslice) * nslice), q2 = q2_lo + (int)(it - row * n2w);
    const int r_lo = slice * rows, nr1 = min(rows, nr1f - r_lo);  // bra entries r_lo .. r_lo + nr1
    // 2 x 2 register tiles of X: rows (r, r + nxr), columns (c, c + nxc), consecutive threads on consecutive c
    const int nxr = (nr1 + 1) >> 1, nxc = (ncd + 1) >> 1;
    const int pr1 = pp_pair[pp1];
    if (same && q2 > pr1 - base1) continue;  // uniform over the block
    const int ij = pp_ij[pp1], a = pair_a[pr1], b = pair_b[pr1];
    const double al = prim_exp[shell_poff[a] + (ij >> 8)], be = prim_exp[shell_poff[b] + (ij & 255)], p = al + be;
    const double ip = 1.0 / p;
    double P[3];
    for (int x = 0; x < 3; ++x) P[x] = (al * shell_xyz[3 * a + x] + be * shell_xyz[3 * b + x]) * ip;
    const int pr2 = base2 + q2, c = pair_a[pr2], d = pair_b[pr2], npd = shell_nprim[d];
    const int npp2 = shell_nprim[c] * npd;
    const double* d2p = dist2 + (pair_ppoff[pr2] - pp_base2) * (int64_t)ncd * nr2;
    __syncthreads();  // the previous item is done with X and the tables
    for (int x = tid; x < nr1 * ncd; x += nth) X[x] = 0.0;
    for (int k0 = 0; k0 < npp2; k0 += chunk) {
      const int nck = min(chunk, npp2 - k0);
      __syncthreads();  // S, F, Z, G of the previous chunk are consumed
      // one thread per ket primitive pair: P - Q, the Boys values, g^{(N)}(u) and u^j
      for (int w = tid; w < nck; w += nth) {
        const int i2 = k0 + w, ic = shell_poff[c] + i2 / npd, id = shell_poff[d] + i2 % npd;
        const double ga = prim_exp[ic], de = prim_exp[id], q = ga + de, iq = 1.0 / q;
        double R[3];
        for (int x = 0; x < 3; ++x) R[x] = P[x] - (ga * shell_xyz[3 * c + x] + de * shell_xyz[3 * d + x]) * iq;
        const double u = R[0] * R[0] + R[1] * R[1] + R[2] * R[2], rpq = 1.0 / (p + q), rho = p * q * rpq;
        for (int x = 0; x < 3; ++x) Rv[3 * w + x] = R[x];
        double* Fw = F + (size_t)w * (lt + 1);
        boys_eval(lt, rho * u, Fw, 1, boys_tab, c_boys);
        // g^{(N)}(u) = 2 pi^{5/2} / (p q sqrt(p + q)) (-rho)^N F_N(rho u), and u^j
        double gN = 2.0 * 5.5683279968317078453 * 3.1415926535897932385 * ip * iq * sqrt(rpq);
        double* Gw = G + (size_t)w * (lt + 1);
        for (int n = 0; n <= lt; ++n) {
          Gw[n] = gN * Fw[n];
          gN *= -rho;
        }
        double* Uw = U + (size_t)w * (lt / 2 + 1);
        double uj = 1.0;
        for (int j = 0; j <= lt / 2; ++j) {
          Uw[j] = uj;
          uj *= u;
        }
      }
      __syncthreads();
      // one thread per (ket primitive pair, harmonic column m) for S_LM(P - Q)
      for (int x = tid; x < nck * (2 * lt + 1); x += nth) {
        const int w = x / (2 * lt + 1), col = x - w * (2 * lt + 1);
        solid_harmonics_columns(lt, Rv[3 * w], Rv[3 * w + 1], Rv[3 * w + 2], S + (size_t)w * nht, col, 2 * lt + 1);
      }
      __syncthreads();
      for (int x = tid; x < nck * nrt; x += nth) {
        const int w = x / nrt, e = x - w * nrt;
        const int r = rmapt[e], h = r & 0xfff, K = r >> 24, L = l_of_index(h);
        const double* Gw = G + (size_t)w * (lt + 1) + L + K;
        const double* Uw = U + (size_t)w * (lt / 2 + 1);
        const double* aK = c2_a + ((size_t)L * (kC2K + 1) + K) * (kC2K + 1);
        double rad = 0.0;
        for (int j = 0; j <= K; ++j) rad = fma(aK[j] * Uw[j], Gw[j], rad);
        // 2^L S_LM(R) rad, the power of two exact
        Z[x] = (S[(size_t)w * nht + h] * rad) * __longlong_as_double((long long)(1023 + L) << 52);
      }
      __syncthreads();
      const int ncol = nck * nr2;  // columns (ket primitive pair, ket entry) of this chunk
      for (int t0 = 0; t0 < ncol; t0 += kEriPartTile) {
        const int tw = min(kEriPartTile, ncol - t0);
        for (int x = tid; x < nr1 * tw; x += nth) {
          const int e1 = x / tw, jj = x - e1 * tw, col = t0 + jj, w = col / nr2, e2 = col - w * nr2;
          const int k1 = kap1[r_lo + e1], k2 = kap2[e2];
          const int h1 = k1 & 0xfff, n1e = (k1 >> 12) & 0xff, L1 = k1 >> 20;
          const int h2 = k2 & 0xfff, n2e = (k2 >> 12) & 0xff, L2 = k2 >> 20;
          const int M1 = h1 - L1 * L1 - L1, M2 = h2 - L2 * L2 - L2;
          const int* lst = L1 >= L2 ? c2_ptr + c2_cbase[L1 * (L1 + 1) / 2 + L2] + (M1 + L1) * (2 * L2 + 1) + M2 + L2
                                    : c2_ptr + c2_cbase[L2 * (L2 + 1) / 2 + L1] + (M2 + L2) * (2 * L1 + 1) + M1 + L1;
          const double* Zw = Z + (size_t)w * nrt;
          double v = 0.0;
          for (int t = lst[0]; t < lst[1]; ++t) {
            const GTerm g = c2_terms[t];
            const int L = g.pad, K = (L1 + L2 - L) / 2 + n1e + n2e;
            v = fma(g.coef, Zw[zoff[L] + (g.ridx - L * L) * (kmax_of(lt, L) + 1) + K], v);
          }
          It[e1 * kEriTileStride + jj] = (L2 & 1) ? -v : v;
        }
        for (int x = tid; x < ncd * tw; x += nth) {
          const int cd = x / tw, jj = x - cd * tw, col = t0 + jj, w = col / nr2, e2 = col - w * nr2;
          Dt[cd * kEriTileStride + jj] = d2p[((int64_t)(k0 + w) * ncd + cd) * nr2 + e2];
        }
        __syncthreads();
        for (int x = tid; x < nxr * nxc; x += nth) {
          const int r0 = x / nxc, c0 = x - r0 * nxc, r1 = r0 + nxr, c1 = c0 + nxc;
          const bool r1ok = r1 < nr1, c1ok = c1 < ncd;
          const double* i0 = It + r0 * kEriTileStride;
          const double* i1 = It + (r1ok ? r1 : r0) * kEriTileStride;
          const double* j0 = Dt + c0 * kEriTileStride;
          const double* j1 = Dt + (c1ok ? c1 : c0) * kEriTileStride;
          double s00 = 0.0, s01 = 0.0, s10 = 0.0, s11 = 0.0;
          for (int jj = 0; jj < tw; ++jj) {
            const double x0 = i0[jj], x1 = i1[jj], y0 = j0[jj], y1 = j1[jj];
            s00 = fma(x0, y0, s00);
            s01 = fma(x0, y1, s01);
            s10 = fma(x1, y0, s10);
            s11 = fma(x1, y1, s11);
          }
          X[r0 * ncd + c0] += s00;
          if (c1ok) X[r0 * ncd + c1] += s01;
          if (r1ok) {
            X[r1 * ncd + c0] += s10;
            if (c1ok) X[r1 * ncd + c1] += s11;
          }
        }
        __syncthreads();
      }
    }
    // this bra primitive pair's and slice's share of the block: D_ab[:, slice] X
    const double* d1 = dist1 + (pp1 - pp_base1) * (int64_t)nab * nr1f + r_lo;
    double* o = part + (row * n2w + (q2 - q2_lo)) * (int64_t)nab * ncd;
    for (int x = tid; x < nab * ncd; x += nth) {
      const int ab = x / ncd, cd = x - ab * ncd;
      const double* dr = d1 + (int64_t)ab * nr1f;
      double s0 = 0.0;
      for (int e1 = 0; e1 < nr1; ++e1) s0 = fma(dr[e1], X[e1 * ncd + cd], s0);
      o[x] = s0;
    }
  }
}

size_t eri_part_smem(int la, int lb, int lc, int ld, int chunk, int nslice) {
  const int lam1 = la + lb, lam2 = lc + ld, lt = lam1 + lam2, nr1 = n_r(lam1), nr2 = n_r(lam2);
  const int rows = (nr1 + nslice - 1) / nslice;
  const size_t ncd = (size_t)(2 * lc + 1) * (2 * ld + 1);
  const size_t dbl = (size_t)rows * ncd + (size_t)rows * kEriTileStride + ncd * kEriTileStride +
                     (size_t)chunk * (n_harm(lt) + 2 * (lt + 1) + n_r(lt) + lt / 2 + 1 + 3);
  return sizeof(double) * dbl + sizeof(int) * (nr1 + nr2 + lt + 1);
}

// Sum of the shares (bra primitive pairs x slices) of each unique quartet (q1 in [q1_lo, q1_hi), q2 in [q2_lo, q2_hi),
// q2 <= q1 for the same class) in a fixed order, written to the eight permutations of every element.  Where
// a = b, c = d or the two pairs coincide the block holds several members of one permutation orbit; only the
// canonical member is written, so the output has the permutational symmetry exactly.  With a density
// (dens != nullptr) every distinct member (pq|rs) of the orbit adds (pq|rs) D_rs to Jm[p][q] and
// (pq|rs) D_qs to Km[p][r] (either may be nullptr); out may then be nullptr.
__global__ void __launch_bounds__(128) k_eri_reduce(int la, int lb, int lc, int ld, int q1_lo, int q1_hi,
                                                    int base1, int q2_lo, int q2_hi, int base2, int same,
                                                    int nslice, int64_t pp_lo, const int* __restrict__ pair_a,
                                                    const int* __restrict__ pair_b,
                                                    const int64_t* __restrict__ pair_ppoff,
                                                    const int* __restrict__ shell_nprim,
                                                    const int64_t* __restrict__ shell_foff,
                                                    const double* __restrict__ part, int64_t nbf,
                                                    double* __restrict__ out, const double* __restrict__ dens,
                                                    double* __restrict__ Jm, double* __restrict__ Km) {
  const int nb = 2 * lb + 1, nd = 2 * ld + 1, nab = (2 * la + 1) * nb, ncd = (2 * lc + 1) * nd;
  const int n2w = q2_hi - q2_lo;
  const int64_t nitems = (int64_t)(q1_hi - q1_lo) * n2w;
  for (int64_t it = blockIdx.x; it < nitems; it += gridDim.x) {
    const int q1 = q1_lo + (int)(it / n2w), q2 = q2_lo + (int)(it - (it / n2w) * n2w);
    if (same && q2 > q1) continue;
    const int pr1 = base1 + q1, pr2 = base2 + q2;
    const int a = pair_a[pr1], b = pair_b[pr1], c = pair_a[pr2], d = pair_b[pr2];
    const int npp1 = shell_nprim[a] * shell_nprim[b] * nslice;  // shares: bra primitive pairs x slices
    const double* src = part + ((pair_ppoff[pr1] - pp_lo) * nslice * n2w + (q2 - q2_lo)) * (int64_t)nab * ncd;
    const int64_t stride = (int64_t)n2w * nab * ncd;
    const int64_t fa = shell_foff[a], fb = shell_foff[b], fc = shell_foff[c], fd = shell_foff[d];
    for (int x = threadIdx.x; x < nab * ncd; x += blockDim.x) {
      const int ab = x / ncd, cd = x - ab * ncd, ma = ab / nb, mb = ab - ma * nb, mc = cd / nd, md = cd - mc * nd;
      if ((a == b && ma < mb) || (c == d && mc < md) || (pr1 == pr2 && ab < cd)) continue;
      double v = 0.0;
      for (int i = 0; i < npp1; ++i) v += src[i * stride + x];
      const int64_t I = fa + ma, J = fb + mb, K = fc + mc, M = fd + md;
      if (out) {
        out[((I * nbf + J) * nbf + K) * nbf + M] = v;
        out[((J * nbf + I) * nbf + K) * nbf + M] = v;
        out[((I * nbf + J) * nbf + M) * nbf + K] = v;
        out[((J * nbf + I) * nbf + M) * nbf + K] = v;
        out[((K * nbf + M) * nbf + I) * nbf + J] = v;
        out[((M * nbf + K) * nbf + I) * nbf + J] = v;
        out[((K * nbf + M) * nbf + J) * nbf + I] = v;
        out[((M * nbf + K) * nbf + J) * nbf + I] = v;
      }
      if (dens) {
        const int64_t t[8][4] = {{I, J, K, M}, {J, I, K, M}, {I, J, M, K}, {J, I, M, K},
                                 {K, M, I, J}, {M, K, I, J}, {K, M, J, I}, {M, K, J, I}};
        for (int u = 0; u < 8; ++u) {
          bool dup = false;
          for (int w = 0; w < u; ++w)
            dup = dup || (t[w][0] == t[u][0] && t[w][1] == t[u][1] && t[w][2] == t[u][2] && t[w][3] == t[u][3]);
          if (dup) continue;
          if (Jm) atomicAdd(Jm + t[u][0] * nbf + t[u][1], v * dens[t[u][2] * nbf + t[u][3]]);
          if (Km) atomicAdd(Km + t[u][0] * nbf + t[u][2], v * dens[t[u][1] * nbf + t[u][3]]);
        }
      }
    }
  }
}

namespace {
// A rectangle of quartets (bra pairs [q1_lo, q1_hi) x ket pairs [q2_lo, q2_hi) of one class pair) whose
// shares fit one stream's scratch region.
struct EriRect {
  int q1_lo, q1_hi, q2_lo, q2_hi;
  int64_t pp_lo, pp_hi;
};

std::vector<EriRect> eri_rects(const ClassWork& w1, const ClassWork& w2, bool same, const int64_t* h_ppoff,
                               int64_t region, int nslice) {
  const int64_t blk = (int64_t)nslice * (2 * w1.la + 1) * (2 * w1.lb + 1) * (2 * w2.la + 1) * (2 * w2.lb + 1);
  const int64_t* pp = h_ppoff + w1.pair_base;  // bra pair q has primitive pairs pp[q] .. pp[q + 1]
  std::vector<EriRect> out;
  int q1 = 0;
  while (q1 < w1.npairs) {
    int q1e = q1 + 1;  // extend the run of bra pairs while the rectangle still fits
    while (q1e < w1.npairs && (pp[q1e + 1] - pp[q1]) * (same ? q1e + 1 : w2.npairs) * blk <= region) ++q1e;
    const int n2 = same ? q1e : w2.npairs;
    if ((pp[q1e] - pp[q1]) * n2 * blk <= region) {
      out.push_back(EriRect{q1, q1e, 0, n2, pp[q1], pp[q1e]});
    } else {  // a single bra pair against too many ket pairs: split the ket range
      const int step = (int)std::max<int64_t>(1, region / ((pp[q1 + 1] - pp[q1]) * blk));
      for (int q2 = 0; q2 < n2; q2 += step)
        out.push_back(EriRect{q1, q1 + 1, q2, std::min(n2, q2 + step), pp[q1], pp[q1 + 1]});
    }
    q1 = q1e;
  }
  return out;
}
}  // namespace

shgo_status launch_eri(const DeviceBasis& db, const DeviceTables& dt, const Tables& th,
                       const std::vector<ClassWork>& work, int64_t nbf, double* out, const double* dens,
                       double* Jm, double* Km, cudaStream_t stream, std::string* err) {
  const size_t nw = work.size();
  std::vector<int64_t> doff(nw + 1, 0);
  for (size_t c = 0; c < nw; ++c) {
    const ClassWork& w = work[c];
    doff[c + 1] = doff[c] + w.npp * (int64_t)(2 * w.la + 1) * (2 * w.lb + 1) * n_r(w.la + w.lb);
  }
  if (doff[nw] == 0) return SHGO_OK;
  ensure_max_dynamic_smem((const void*)k_eri_part);
  // class pairs, largest first, and each one's chunk of ket primitive pairs
  struct CP {
    size_t c1, c2;
    double cost;
    int chunk, nslice;
  };
  std::vector<CP> cps;
  int64_t need_max = 0, one_max = 1;
  for (size_t c1 = 0; c1 < nw; ++c1)
    for (size_t c2 = 0; c2 <= c1; ++c2) {
      const ClassWork &w1 = work[c1], &w2 = work[c2];
      if (w1.npairs == 0 || w2.npairs == 0) continue;
      const double nq = c1 == c2 ? 0.5 * w1.npp * (w1.npairs + 1) : (double)w1.npp * w2.npairs;
      const double ppq = nq * ((double)w2.npp / w2.npairs);
      const double cost = ppq * n_r(w1.la + w1.lb) * n_r(w2.la + w2.lb) * (2 * w2.la + 1) * (2 * w2.lb + 1);
      int maxnp = 1;
      for (int q = 0; q < w2.npairs; ++q)
        maxnp = (int)std::max<int64_t>(maxnp, db.h_ppoff[w2.pair_base + q + 1] - db.h_ppoff[w2.pair_base + q]);
      // shared memory within kEriSmemTarget (four blocks of 256 threads per SM): fewer ket primitive pairs per
      // chunk first, then the bra entries cut into slices
      int chunk = std::min(16, maxnp), nslice = 1;
      while (chunk > 1 && eri_part_smem(w1.la, w1.lb, w2.la, w2.lb, chunk, 1) > kEriSmemTarget) --chunk;
      while (nslice < n_r(w1.la + w1.lb) && eri_part_smem(w1.la, w1.lb, w2.la, w2.lb, chunk, nslice) > kEriSmemTarget)
        ++nslice;
      cps.push_back(CP{c1, c2, cost, chunk, nslice});
      const int64_t full = (c1 == c2 ? w1.npp * (int64_t)w1.npairs : w1.npp * (int64_t)w2.npairs) * nslice *
                           (2 * w1.la + 1) * (2 * w1.lb + 1) * (2 * w2.la + 1) * (2 * w2.lb + 1);
      need_max = std::max(need_max, full);
      int64_t np1 = 1;  // one bra pair against one ket pair must fit a region
      for (int q = 0; q < w1.npairs; ++q)
        np1 = std::max<int64_t>(np1, db.h_ppoff[w1.pair_base + q + 1] - db.h_ppoff[w1.pair_base + q]);
      one_max = std::max(one_max, np1 * nslice * (2 * w1.la + 1) * (2 * w1.lb + 1) * (2 * w2.la + 1) * (2 * w2.lb + 1));
    }
  std::stable_sort(cps.begin(), cps.end(), [](const CP& x, const CP& y) { return x.cost > y.cost; });
  cudaStream_t* pool = nullptr;
  cudaError_t e = stream_pool(&pool);
  if (e != cudaSuccess) {
    *err = std::string("stream pool: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  const int ns = (int)std::min<size_t>(cps.size(), (size_t)kPoolStreams);
  // scratch region per stream: what the largest class pair needs, at most 8M doubles (64 MiB) unless
  // SHGO_ERI_SCRATCH_DOUBLES sets another cap; never less than one bra pair against one ket pair
  int64_t cap = (int64_t)1 << 23;
  if (const char* env = std::getenv("SHGO_ERI_SCRATCH_DOUBLES")) {
    const long long v = std::atoll(env);
    if (v > 0) cap = v;
  }
  const int64_t region = std::max<int64_t>(std::min<int64_t>(need_max, cap), one_max);
  double* dist = nullptr;
  e = workspace_alloc((void**)&dist, sizeof(double) * (size_t)(doff[nw] + (int64_t)ns * region), stream);
  if (e != cudaSuccess) {
    *err = std::string("distribution and scratch buffers: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? SHGO_ERR_OOM : SHGO_ERR_CUDA;
  }
  double* scratch = dist + doff[nw];
  for (size_t c = 0; c < nw; ++c) {
    const ClassWork& w = work[c];
    if (w.npp == 0) continue;
    const int cid = class_id(w.la, w.lb);
    k_eri_dist<<<grid_cap(w.npp, 8), 128, eri_dist_smem(w.la, w.lb), stream>>>(
        w.la, w.lb, w.npp, w.pp_base, db.pp_pair, db.pp_ij, db.pair_a, db.pair_b, db.shell_xyz, db.shell_poff,
        db.prim_exp, db.prim_coef, dt.etab, dt.eoff, dt.gt_ptr + th.gt_base[cid], dt.gt_terms + th.gt_termbase[cid],
        dt.eri_eps, dist + doff[c]);
  }
  cudaEvent_t fork;
  e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    cudaFreeAsync(dist, stream);
    *err = std::string("fork event: ") + cudaGetErrorString(e);
    return SHGO_ERR_CUDA;
  }
  bool joined = true;
  {
    cudaEventRecord(fork, stream);
    for (int i = 0; i < ns; ++i) cudaStreamWaitEvent(pool[i], fork, 0);
    for (size_t k = 0; k < cps.size(); ++k) {
      const ClassWork &w1 = work[cps[k].c1], &w2 = work[cps[k].c2];
      const bool same = cps[k].c1 == cps[k].c2;
      cudaStream_t s = pool[k % ns];
      double* reg = scratch + (int64_t)(k % ns) * region;
      const int lam1 = w1.la + w1.lb, lam2 = w2.la + w2.lb;
      const int nsl = cps[k].nslice;
      // threads per block: fewer for the small class pairs, so that more items are resident per SM
      const int xw = ((n_r(lam1) + nsl - 1) / nsl) * (2 * w2.la + 1) * (2 * w2.lb + 1);
      const int threads = xw >= 1024 ? 256 : (xw >= 256 ? 128 : 64);
      for (const EriRect& r : eri_rects(w1, w2, same, db.h_ppoff, region, nsl)) {
        const int64_t items = (r.pp_hi - r.pp_lo) * nsl * (int64_t)(r.q2_hi - r.q2_lo);
        // one block per item, so that blocks of the class pairs running on other streams share the SMs
        k_eri_part<<<(unsigned)std::min<int64_t>(items, 0x7fffffff), threads,
                     eri_part_smem(w1.la, w1.lb, w2.la, w2.lb, cps[k].chunk, nsl), s>>>(
            w1.la, w1.lb, w2.la, w2.lb, r.pp_lo, r.pp_hi, w1.pair_base, r.q2_lo, r.q2_hi, same ? 1 : 0,
            cps[k].chunk, nsl, db.pp_pair, db.pp_ij, db.pair_a, db.pair_b, db.pair_ppoff, w1.pp_base, w2.pp_base,
            w2.pair_base, db.shell_xyz, db.shell_poff, db.shell_nprim, db.prim_exp, dist + doff[cps[k].c1],
            dist + doff[cps[k].c2], dt.boys, dt.rmap + th.rmap_off[lam1], dt.rmap + th.rmap_off[lam2],
            dt.rmap + th.rmap_off[lam1 + lam2], dt.c2_ptr, dt.c2_cbase, dt.c2_terms, dt.c2_a, reg);
        const int64_t quartets = (int64_t)(r.q1_hi - r.q1_lo) * (r.q2_hi - r.q2_lo);
        k_eri_reduce<<<grid_cap(quartets, 16), 128, 0, s>>>(
            w1.la, w1.lb, w2.la, w2.lb, r.q1_lo, r.q1_hi, w1.pair_base, r.q2_lo, r.q2_hi, w2.pair_base,
            same ? 1 : 0, nsl, r.pp_lo, db.pair_a, db.pair_b, db.pair_ppoff, db.shell_nprim, db.shell_foff, reg, nbf, out,
            dens, Jm, Km);
      }
    }
    for (int i = 0; i < ns && joined; ++i) {
      cudaEvent_t join;
      if (cudaEventCreateWithFlags(&join, cudaEventDisableTiming) != cudaSuccess) {
        joined = false;
        break;
      }
      cudaEventRecord(join, pool[i]);
      cudaStreamWaitEvent(stream, join, 0);
      cudaEventDestroy(join);
    }
    cudaEventDestroy(fork);
  }
  shgo_status st = launch_error(err);
  if (!joined) {
    // `stream` does not wait for every pool stream: finish their work before the buffers are returned
    for (int i = 0; i < ns; ++i) cudaStreamSynchronize(pool[i]);
    if (st == SHGO_OK) {
      st = SHGO_ERR_CUDA;
      *err = "join event could not be created";
    }
  }
  cudaFreeAsync(dist, stream);
  return st;
}

cudaError_t ensure_max_dynamic_smem(const void* func, int bytes) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> done;  // (kernel, device) pairs already set
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  for (const auto& d : done)
    if (d.first == func && d.second == dev) return cudaSuccess;
  e = bytes > 0 ? cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
                : set_max_dynamic_smem(func);
  if (e == cudaSuccess) done.emplace_back(func, dev);
  return e;
}

int64_t launches_per_call(const std::vector<ClassWork>& work, int64_t nbf) {
  int64_t n = 0;
  for (const auto& w : work) n += (w.npp > 0 ? 1 : 0) + (w.npairs > 0 ? 1 : 0);
  return nbf == 0 ? 0 : n;
}

}  // namespace shgo
