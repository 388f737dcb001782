// Adjoint of the ray trace: gradients of L = sum_p w_p Gamma_p with respect to
// log n_HI of every cell and log Ndot of every source.
//
// The forward recurrence of one (source, face) item (trace.cu) is
//   tau_in(p)  = sum_n w_n(p) tau_out(e_n(p))      (m >= 2; m = 1: dtau(s)/2 ds(p))
//   tau_out(p) = tau_in(p) + dtau(p) ds(p)
//   Gamma_sp   = Ndot [g(tau_in) - g(tau_out)] / (n_HI V)  or  Ndot sigma0 h(tau_in)/(4 pi r^2)
// so with lambda(p) = dL/dtau_out(p) and mu(p) = dL/dtau_in(p):
//   lambda(p) = w_p dGamma_sp/dtau_out + sum_{q uses p} w_n(q) mu(q)
//   mu(p)     = lambda(p) + w_p dGamma_sp/dtau_in        (rates: in the reverse pass only)
//   dL/dlog n_HI(p) += dtau(p) ds(p) lambda(p) - w_p Gamma_sp   (the last term: thick, 1/n_HI)
//   dL/ddtau(s)     += sum_{m=1 cells} mu(p) ds(p)/2 + lambda(s)/2
//   dL/dlog Ndot_s   = sum_p w_p Gamma_sp                         (Gamma is linear in Ndot)
// The users q of p lie in the next layer of the same face.  Each face seeds
// the adjoint with the direct terms of the cells it owns and propagates it
// through its whole closed pyramid, which contains the complete upstream cone
// of every cell in it; summing the faces' partial adjoints gives the total.
//
// Items are (source, face, quadrant) as in the batched trace.  Per item: a
// forward pass stores (tau_in, tau_out) of every layer in a per-CTA stack in
// global memory (the per-source column densities are never
// kept beyond the item), then a reverse pass walks the layers from the outside
// in with mu of the next layer in shared memory.  Built with --fmad=false.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "asora_internal.cuh"
#include "device_util.cuh"
#include "faces.cuh"

namespace asora {

// Stack capacity (double2) of one quadrant item for radius limit r2, box size n.
size_t face_stack_cap(int r2, int nmax) {
  size_t tot = 0;
  int L = (int)std::floor(std::sqrt((double)r2));
  while ((int64_t)L * L > r2) --L;
  L = std::min(L, nmax / 2 + 1);
  for (int m = 1; m <= L; ++m) {
    int h = (int)std::floor(std::sqrt((double)(r2 - m * m)));
    while (h > 0 && (int64_t)h * h > r2 - (int64_t)m * m) --h;
    h = std::min(h, m);
    tot += (size_t)(h + 1) * (h + 1);
  }
  return tot;
}

__host__ __device__ inline size_t r16(size_t x) { return (x + 15) & ~(size_t)15; }

// Shared memory of one adjoint group: two layers of (h+1)^2 doubles, one row
// table (h+2 ints, (h+1)^2 bytes), per-layer metadata (half-width, stack
// offset, "has rate cells" flag) for lcap layers, reduction scratch.
__host__ __device__ inline size_t bwd_group_bytes(int h, int lcap) {
  const size_t cap = (size_t)(h + 1) * (h + 1);
  return r16(2 * cap * sizeof(double)) + r16((size_t)(h + 2) * sizeof(int)) + r16(cap) +
         r16(2 * (size_t)(lcap + 2) * sizeof(int)) + r16((size_t)(lcap + 2)) + 64;
}

size_t bwd_smem_bytes(int hcap, int lcap) { return bwd_group_bytes(hcap, lcap); }

struct BwdArgs {
  TraceArgs t;
  const double* w;       // dL/dGamma per cell
  double* dlogn;         // dL/dlog n_HI per cell (accumulated)
  double* dndot;         // dL/dlog Ndot per merged source (accumulated)
  double2* stack;        // per-group (tau_in, tau_out) stacks
  size_t stack_cap;      // double2 per group
  int lcap;              // layer capacity of the metadata arrays
  int exit;              // stop the recompute at the first opaque layer (exact)
  // faces by warps (k_bwd_faces): quadrant items of the faces it could not finish, those
  // of sources before split_src from redo[0] on, the others from redo[redo_cap] on
  int* redo;
  int* redo_n;
  int redo_cap, split_src;
  const int* n_dev;      // quadrant kernels: number of items, if it is on the device
};

template <int GS>
__device__ __forceinline__ bool group_any(bool v) {
  if (GS == 32) {
    __syncwarp();
    return __any_sync(0xffffffffu, v);
  }
  return __syncthreads_or(v) != 0;
}

template <int GS>
__device__ __forceinline__ bool group_all(bool v) {
  if (GS == 32) {
    __syncwarp();
    return __all_sync(0xffffffffu, v);
  }
  return __syncthreads_and(v) != 0;
}

// Sum over the group; the result is valid in thread 0 of the group.
template <int GS>
__device__ __forceinline__ double group_sum(double v, double* red, int gt) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (GS == 32) return v;
  group_sync<GS>();
  if ((gt & 31) == 0) red[gt >> 5] = v;
  group_sync<GS>();
  double s = 0.0;
  if (gt == 0)
    for (int i = 0; i < GS / 32; ++i) s += red[i];
  return s;
}

// Direct terms of an owned cell with a rate and w != 0: adds w Gamma to qacc and returns
// dL/dtau_in; lam (in: what arrives from the cell's users) becomes dL/dtau_out, ndir the
// 1/n_HI term of dL/dlog n_HI.  In the thick form the two derivatives combine as the slope
// difference g'(tau_in) - g'(tau_out) (0 within one chord segment) before adding.
// FP64 issue binds the reverse pass, and a predicated-off FP64 instruction takes its full
// turn: zero tests are integer ones, products are formed once and fused, and the thin
// form is out of line.
struct ThinTerms {
  double wG, dmu;
};
__device__ __noinline__ ThinTerms thin_terms(const double2* __restrict__ htab, const TabDev* tab,
                                             double wf, double tin) {
  return {wf * tab_eval(htab, *tab, tin), wf * tab_slope(htab, *tab, tin)};
}

__device__ __forceinline__ double direct_terms(const TraceArgs& a, const double nd_thick,
                                               const double nd_thin, const double2 gv,
                                               const double* invn, const double wp,
                                               const double dtp, const double dcell,
                                               const double tin, const double tout, double& lam,
                                               double& ndir, double& qacc) {
  bool thin = __double2hiint(dtp) <= __double2hiint(a.tau_lim);  // (ds >= 1)
  if (thin) thin = bits_of(dcell) <= bits_of(a.tau_lim);
  double mup;
  if (thin) {
    const ThinTerms t = thin_terms(a.tab.h, &a.tab, wp * (nd_thin * gv.y), tin);
    qacc += t.wG;
    mup = lam + t.dmu;
  } else {
    const double wf = wp * (nd_thick * (gv.x * __ldg(invn)));
    const double wG = wf * (tab_eval(a.tab.g, a.tab, tin) - tab_eval(a.tab.g, a.tab, tout));
    const double si = tab_slope(a.tab.g, a.tab, tin), so = tab_slope(a.tab.g, a.tab, tout);
    qacc += wG;
    mup = fma(wf, si - so, lam);
    lam = fma(-wf, so, lam);
    ndir = -wG;
  }
  return mup;
}

// One (source, face, quadrant) item of the adjoint with a group of GS threads.
template <int GS>
__device__ __forceinline__ void bwd_item(const BwdArgs& A, const int item, const int gt,
                                         unsigned char* __restrict__ sm, double2* __restrict__ stk) {
  const TraceArgs& a = A.t;
  const int h = a.hcap;
  const int cap = (h + 1) * (h + 1);
  double* bufA = reinterpret_cast<double*>(sm);
  double* bufB = bufA + cap;
  unsigned char* p = sm + r16(2 * (size_t)cap * sizeof(double));
  int* rowpre = reinterpret_cast<int*>(p);
  p += r16((size_t)(h + 2) * sizeof(int));
  unsigned char* rowof = p;
  p += r16((size_t)cap);
  int* lH = reinterpret_cast<int*>(p);
  int* lO = lH + A.lcap + 2;
  p += r16(2 * (size_t)(A.lcap + 2) * sizeof(int));
  unsigned char* lnear = p;
  p += r16((size_t)(A.lcap + 2));
  double* red = reinterpret_cast<double*>(p);
  const int wid = gt >> 5, lane = gt & 31;

  const int s = item >> 5, f = (item >> 2) & 7, quad = item & 3;
  const SrcDev S = a.src[s];
  const BoxDev B = a.boxes[S.box];
  const int N = B.n;
  const int R2 = a.r2lim[s];
  const double nd = a.ndot[s];
  const int d = f >> 1;
  const int sg = (f & 1) ? -1 : 1;
  const int q1 = (quad & 1) ? -1 : 1, q2 = (quad & 2) ? -1 : 1;
  const int lim1 = q1 > 0 ? B.whi : -B.wlo, lim2 = q2 > 0 ? B.whi : -B.wlo;
  int Lmax = sg > 0 ? B.whi : -B.wlo;
  Lmax = min(Lmax, isqrt_i(R2));
  if (Lmax > A.lcap) {
    if (gt == 0) atomicOr(a.err, ERR_LAYER_CAP);
    return;
  }
  const int64_t scell = B.off + ((int64_t)S.i * N + S.j) * N + S.k;
  const double dts = a.dtau[scell];
  const int64_t NN = (int64_t)N * N;
  const int c1 = d == 0 ? S.j : S.i;
  const int c2 = d == 2 ? S.j : S.k;
  const int cd = d == 0 ? S.i : (d == 1 ? S.j : S.k);
  const int64_t m1 = d == 0 ? (int64_t)N : (d == 1 ? NN : (int64_t)N);
  const int64_t md = d == 0 ? NN : (d == 1 ? (int64_t)N : NN);
  const double* __restrict__ fld = (d == 2 ? a.dtauT : a.dtau) + B.off;
  const double nd_thick = nd * B.inv_cell3, nd_thin = nd * B.thin_fac;
  double qacc = 0.0;    // sum_p w_p Gamma_sp over owned cells of this item
  double srcacc = 0.0;  // dL/ddtau(s) from this item

  // source cell (owned by face 4, quadrant 0): rate, its Ndot and tau_out adjoints
  double lam_s = 0.0, ndir_s = 0.0;
  if (f == 4 && quad == 0 && gt == 0) {
    const double tout = 0.5 * dts;
    const double ws = A.w[scell];
    if (bits_of(tout) <= bits_of(a.tau_lim)) {
      qacc += ws * (nd * (tab_eval(a.tab.h, a.tab, 0.0) * (0.5 * B.thin_fac)));
    } else {
      const double fct = nd * B.inv_cell3 * a.invn[scell];
      const double G = fct * (tab_eval(a.tab.g, a.tab, 0.0) - tab_eval(a.tab.g, a.tab, tout));
      qacc += ws * G;
      lam_s = -ws * fct * tab_slope(a.tab.g, a.tab, tout);
      ndir_s = -ws * G;
    }
  }

  // ------------------------------------------------ forward (recompute)
  double* prev = bufA;
  double* cur = bufB;
  int Hp = 0, Llast = 0;
  size_t off = 0;
  if (gt == 0) prev[0] = 0.5 * dts;  // the interpolant of every layer-1 cell
  for (int m = 1; m <= Lmax; ++m) {
    const int rem = R2 - m * m;
    const int H = min(m, isqrt_i(rem));
    const size_t W2 = (size_t)(H + 1) * (H + 1);
    if (H > h || m > a.kap_mmax || off + W2 > A.stack_cap) {
      if (gt == 0) atomicOr(a.err, ERR_LAYER_CAP);
      return;
    }
    if (gt == 0) {
      lH[m] = H;
      lO[m] = (int)off;
    }
    const int nrows = min(H, lim1) + 1;
    if (wid == 0) quad_rows_warp(rem, H, nrows, lim2, rowpre, rowof, lane);
    group_sync<GS>();
    const int total = rowpre[nrows];
    const int W = H + 1, Wp = Hp + 1;
    const int lc = wrapc(cd + sg * m, N);
    const int64_t lay = (int64_t)lc * md;
    const int gbase = (int)geo_index(m, 0, 0);
    bool near = false, opaque = true;
    for (int t = gt; t < total; t += GS) {
      const int a1 = rowof[t];
      const int a2 = t - rowpre[a1];
      const int x1 = wrapc(c1 + q1 * a1, N), x2 = wrapc(c2 + q2 * a2, N);
      const int64_t gidx = lay + x1 * m1 + x2;
      const double dtp = __ldg(&fld[gidx]);
      const GeoEntry* ge = &a.geo[gbase + ((max(a1, a2) * (max(a1, a2) + 1)) >> 1) + min(a1, a2)];
      const double ds = __ldg(&ge->ds);
      // Layer 1 (tau_in = (dtau_s/2) ds) goes through the same chain, so that no
      // branch on m turns into an FP64 product issued with every lane predicated
      // off in the other layers' rounds: its interpolants all read slot 0 of the
      // previous buffer, which holds dtau_s/2, with weights (ds, 0, 0, 0); the
      // zero terms add exactly +0.
      const bool l1 = m == 1;
      const double wa = __ldg(&ge->wa), wb = __ldg(&ge->wb);
      const double w1 = l1 ? ds : __ldg(&ge->w1), w4 = l1 ? 0.0 : __ldg(&ge->w4);
      const double w2 = l1 ? 0.0 : (a1 <= a2 ? wa : wb);
      const double w3 = l1 ? 0.0 : (a1 <= a2 ? wb : wa);
      const int b1 = min(a1, Hp), b2 = min(a1 - (a1 > 0), Hp);
      const int e1 = min(a2, Hp), e2 = min(a2 - (a2 > 0), Hp);
      const double tin = fma(w4, prev[b2 * Wp + e2],
                             fma(w3, prev[b1 * Wp + e2], fma(w2, prev[b2 * Wp + e1],
                                                             w1 * prev[b1 * Wp + e1])));
      const double tout = fma(dtp, ds, tin);
      const int li = a1 * W + a2;
      cur[li] = tout;
      stk[off + li] = make_double2(tin, tout);
      opaque = opaque && bits_of(tout) >= a.exit_bits;
      const bool rate = bits_of(tin) < a.tab.tau_max_bits;
      near = near || rate;
    }
    const bool near_any = group_any<GS>(near);
    const bool all_opaque = group_all<GS>(opaque);
    if (gt == 0) lnear[m] = near_any ? 1 : 0;
    double* tmp = prev;
    prev = cur;
    cur = tmp;
    Hp = H;
    off += W2;
    Llast = m;
    // No rate beyond a fully opaque layer (every later tau_in >= 2^E1): the
    // adjoint gets nothing from the rest of the pyramid.
    if (A.exit && all_opaque) break;
  }
  group_sync<GS>();

  // ------------------------------------------------ reverse
  double* next = bufA;  // mu of layer m+1
  double* mu = bufB;    // mu of layer m
  int Hn = -1;
  bool nz_next = false;  // whether layer m+1 has any non-zero mu
  for (int m = Llast; m >= 1; --m) {
    const int H = lH[m];
    if (!nz_next && !lnear[m]) {
      // no adjoint arrives and no rate cell: mu = 0 and nothing to deposit here
      Hn = H;
      continue;
    }
    const int rem = R2 - m * m;
    const int W = H + 1, Wn = Hn + 1;
    for (int t = gt; t < W * W; t += GS) mu[t] = 0.0;
    const int nrows = min(H, lim1) + 1;
    if (wid == 0) quad_rows_warp(rem, H, nrows, lim2, rowpre, rowof, lane);
    group_sync<GS>();
    const int total = rowpre[nrows];
    const int lc = wrapc(cd + sg * m, N);
    const int64_t lay = (int64_t)lc * md;
    const int gbase = (int)geo_index(m, 0, 0);
    const size_t o = (size_t)lO[m];
    bool nz = false;
    for (int t = gt; t < total; t += GS) {
      const int a1 = rowof[t];
      const int a2 = t - rowpre[a1];
      const int li = a1 * W + a2;
      // users of p in layer m+1 of this quadrant: (a1 | a1+1, a2 | a2+1); with M =
      // mu / kappa their weights are all one (see bwd_face)
      double lam = 0.0;
      const int go = (int)georow_index(m, 0, 0) + a1 * (m + 1) + a2;
      if (nz_next) {
        const double* q = next + a1 * Wn + a2;
        const bool u0 = a1 <= Hn, u1 = a1 < Hn, v0 = a2 <= Hn, v1 = a2 < Hn;
        lam = __ldg(&a.kappa[go]) * (((u0 && v0 ? q[0] : 0.0) + (u1 && v0 ? q[Wn] : 0.0)) +
                                     ((u0 && v1 ? q[1] : 0.0) + (u1 && v1 ? q[Wn + 1] : 0.0)));
      }
      double2 tt = make_double2(0.0, 0.0);
      bool rate = false;
      if (lnear[m]) {
        tt = stk[o + li];
        rate = bits_of(tt.x) < a.tab.tau_max_bits;
      }
      if (!nonzero(lam) && !rate) continue;  // mu = 0 (zeroed) and nothing to deposit
      const double tin = tt.x, tout = tt.y;
      const bool own = ((d == 2) || (d == 1 ? a2 < m : (a1 < m && a2 < m))) &&
                       (a1 > 0 || q1 > 0) && (a2 > 0 || q2 > 0);
      const int x1 = wrapc(c1 + q1 * a1, N), x2 = wrapc(c2 + q2 * a2, N);
      const int64_t gidx = lay + x1 * m1 + x2;
      const int64_t cell = B.off + (d == 2 ? ((int64_t)x1 * N + x2) * N + lc : gidx);
      const GeoEntry* ge = &a.geo[gbase + ((max(a1, a2) * (max(a1, a2) + 1)) >> 1) + min(a1, a2)];
      const double ds = __ldg(&ge->ds);
      const double dtp = __ldg(&fld[gidx]);
      double mup = lam, ndir = 0.0;
      const double dcell = dtp * ds;
      const double wp = own && rate ? __ldg(&A.w[cell]) : 0.0;
      if (nonzero(wp))
        mup = direct_terms(a, nd_thick, nd_thin, make_double2(__ldg(&ge->invv), __ldg(&ge->thin)),
                           &a.invn[cell], wp, dtp, dcell, tin, tout, lam, ndir, qacc);
      const double contrib = fma(dcell, lam, ndir);
      nz = nz || nonzero(mup);
      mu[li] = mup * __ldg(&a.ikappa[go]);
      if (nonzero(contrib)) atomicAdd(&A.dlogn[cell], contrib);
    }
    if (m == 1) {
      // dL/ddtau(s) from layer 1, after its rounds (kept out of the cell loop so that
      // no FP64 product runs with every lane off in the other layers): the same
      // thread takes the same cells as in the loop, so each partial sum is unchanged
      for (int t = gt; t < total; t += GS) {
        const int a1 = rowof[t];
        const int a2 = t - rowpre[a1];
        const GeoEntry* ge = &a.geo[gbase + ((max(a1, a2) * (max(a1, a2) + 1)) >> 1) + min(a1, a2)];
        const double mup = mu[a1 * W + a2];  // (kappa = 1 in layer 1)
        if (!nonzero(mup)) continue;  // mu = 0: no term (as in the loop)
        srcacc += mup * (0.5 * __ldg(&ge->ds));
      }
    }
    nz_next = group_any<GS>(nz);
    double* tmp = next;
    next = mu;
    mu = tmp;
    Hn = H;
  }
  // per-item reductions: dL/dlog Ndot and the source cell's dtau adjoint
  const double qsum = group_sum<GS>(qacc, red, gt);
  const double ssum = group_sum<GS>(srcacc, red, gt);
  if (gt == 0) {
    if (qsum != 0.0) atomicAdd(&A.dndot[s], qsum);
    const double cs = dts * (ssum + 0.5 * lam_s) + ndir_s;
    if (cs != 0.0) atomicAdd(&A.dlogn[scell], cs);
  }
  group_sync<GS>();
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 6) k_trace_faces_bwd(BwdArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  const TraceArgs& a = A.t;
  if (a.skip && *a.skip) return;
  double2* stk = A.stack + (size_t)blockIdx.x * A.stack_cap;
  const int cap = (a.hcap + 1) * (a.hcap + 1);
  double* buf = reinterpret_cast<double*>(smem_raw);
  for (int t = threadIdx.x; t < 2 * cap; t += BLOCK) buf[t] = 0.0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = a.item_begin + atomicAdd(a.queue, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= (A.n_dev ? *A.n_dev : a.n_items)) break;
    bwd_item<BLOCK>(A, a.items[it], threadIdx.x, smem_raw, stk);
  }
}

template <int WPB>
__global__ void __launch_bounds__(WPB * 32, 2) k_trace_faces_bwd_warp(BwdArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TraceArgs& a = A.t;
  if (a.skip && *a.skip) return;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* my = smem_raw + (size_t)wid * bwd_group_bytes(a.hcap, A.lcap);
  double2* stk = A.stack + ((size_t)blockIdx.x * WPB + wid) * A.stack_cap;
  const int cap = (a.hcap + 1) * (a.hcap + 1);
  double* buf = reinterpret_cast<double*>(my);
  for (int t = lane; t < 2 * cap; t += 32) buf[t] = 0.0;
  __syncwarp();
  for (;;) {
    int it = 0;
    if (lane == 0) it = a.item_begin + atomicAdd(a.queue, 1);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= (A.n_dev ? *A.n_dev : a.n_items)) break;
    bwd_item<32>(A, a.items[it], lane, my, stk);
  }
}

// ------------------------------------------------------------ whole faces
// The adjoint of one face by one warp.  The recompute of nearly every item ends after a
// few layers, at the first opaque one, so what an item costs is latency: a face at once
// takes a quarter of the steps and of the per-layer work of its four quadrants, its cells
// come from the face tables of rates.cu, in one layer buffer updated in place, and the
// rate and its derivatives are evaluated in the reverse pass only.
// With M = mu / kappa (rates.cu: kappa = C(m, |t1|) C(m, |t2|)) the weights of the users
// of a cell are all one: lambda = kappa (sum of M over its users) + direct terms.  The
// reverse pass takes the cells inside out: a cell reads its own slot and those further
// out, none of which has been rewritten.  Slots outside layer m + 1 are zero (layers
// shrink outwards, so whatever wrote them is also a user).
// A face with a layer wider than the buffer (h), before it is opaque or ends, is left to
// the quadrant kernels.
//
// On an axis the outward step goes to either side: the terms that the four of a cell off
// the axes do not cover (out of line, see direct_terms).
__device__ __noinline__ double axis_users(const double* s, double sum, int W, int t1, int t2) {
  if (t1 == 0) {
    const int d2 = t2 < 0 ? -1 : 1;
    sum += s[-W] + s[-W + d2];
    if (t2 == 0) sum += s[-1] + (s[W - 1] + s[-W - 1]);
  } else if (t2 == 0) {
    const int d1 = t1 < 0 ? -W : W;
    sum += s[-1] + s[d1 - 1];
  }
  return sum;
}

__device__ __forceinline__ void bwd_face(const BwdArgs& A, const int item, const int lane,
                                         unsigned char* __restrict__ sm,
                                         double2* __restrict__ stk) {
  constexpr unsigned FULL = 0xffffffffu;
  const TraceArgs& a = A.t;
  const int h = a.hcap;
  const int W = 2 * h + 3;
  const int TS = face_slot_bytes(h);
  double* buf = reinterpret_cast<double*>(sm);
  double* const org = buf + (h + 1) * (W + 1);
  unsigned char* tab = sm + face_layer_bytes(h);
  const Quad Q = quad_setup(a, item);
  const int s = item >> 5;
  const int hz = min(h, isqrt_i(Q.R2 >> 1));
  auto clear = [&]() {  // every slot that a cell or its neighbours use, and the zero slot
    for (int t = (h - hz) * W + lane; t < (h + hz + 3) * W; t += 32) buf[t] = 0.0;
    if (lane == 0) buf[0] = 0.0;
  };
  clear();
  const int ent = first_layer_entry(a, Q.R2, 1 << 30);
  auto layer = [&](int m) { return __ldg(&a.ftab_lay[ent + m - 1]); };
  auto fits = [&](const int4& l, size_t off) {
    return l.y > 0 && l.y <= TS && l.w <= h && off + l.z <= A.stack_cap;
  };
  auto stage = [&](int m, const int4& l) {
    stage_rows<32>(a.ftab + l.x, l.y, tab + (m & 1) * TS, lane);
  };
  auto cells_of = [&](int m) { return reinterpret_cast<const char2*>(tab + (m & 1) * TS); };
  auto base_of = [&](int m) { return wrapc(Q.cd + Q.sg * m, Q.N) * Q.md + Q.org; };
  auto in_window = [&](const CellIn& c) { return c.t1 <= Q.lim1 && c.t2 <= Q.lim2; };

  // ------------------------------------------------ forward (recompute)
  int Llast = 0;
  unsigned near_bits = 0;  // layers with a cell that can have a rate
  size_t off = 0;
  bool cut = ent < 0 && Q.Lmax >= 1;
  if (!cut && Q.Lmax >= 1) {
    int4 cur = layer(1), nxt = Q.Lmax > 1 ? layer(2) : make_int4(0, 0, 0, 0);
    cut = !fits(cur, 0);
    if (!cut) stage(1, cur);
    for (int m = 1; !cut && m <= Q.Lmax; ++m) {
      cp_async_wait_all();
      __syncwarp();
      const bool go_on = m < Q.Lmax && m < 31 && m < a.kap_mmax && fits(nxt, off + cur.z);
      int4 nn = make_int4(0, 0, 0, 0);
      if (go_on) {
        stage(m + 1, nxt);
        if (m + 2 <= Q.Lmax) nn = layer(m + 2);
      }
      const char2* cells = cells_of(m);
      const int base = base_of(m);
      const GeoRow* grow = a.georow + georow_index(m, 0, 0);
      bool near = false, opaque = true;
      CellIn nc;
      Weights nw;
      auto load = [&](int t) {
        fetch_face_cell(Q, nc, max(t, 0), base, cells);
        nw = load_weights(grow + abs(nc.t1) * (m + 1) + abs(nc.t2));
      };
      load(cur.z - 1 - lane);
      auto step = [&](int T, auto first) {
        constexpr bool FIRST = decltype(first)::value;
        const CellIn c = nc;
        const Weights w = nw;
        if (T >= 32) load(T - 32 - lane);
        double* sc = org + c.t1 * W + c.t2;
        double tin;
        if constexpr (FIRST) tin = Q.half_dts * w.ds;  // source centre to the entry plane
        else tin = interp(a, w, sc, sgn_i(c.t1) * W, sgn_i(c.t2));
        const double tout = fma(c.dtp, w.ds, tin);
        __syncwarp();  // all reads before any write
        if (T - lane >= 0) {
          stk[off + T - lane] = make_double2(tin, tout);
          if (in_window(c)) {
            *sc = tout;
            opaque = opaque && bits_of(tout) >= a.exit_bits;
            near = near || bits_of(tin) < a.tab.tau_max_bits;
          }
        }
        __syncwarp();
      };
      if (m == 1) step(cur.z - 1, std::true_type());  // (at most nine cells)
      else
        for (int T = cur.z - 1; T >= 0; T -= 32) step(T, std::false_type());
      if (__any_sync(FULL, near)) near_bits |= 1u << m;
      Llast = m;
      off += cur.z;
      if (A.exit && __all_sync(FULL, opaque)) break;
      cut = m < Q.Lmax && !go_on;
      cur = nxt;
      nxt = nn;
    }
    cp_async_wait_all();
    __syncwarp();
  }
  if (cut && !A.redo_cap) {  // (the host gives every face that may be cut a place)
    if (lane == 0) atomicOr(a.err, ERR_LAYER_CAP);
    return;
  }
  if (cut) {
    const int kind = s < A.split_src ? 0 : 1;
    int at = 0;
    if (lane == 0) at = atomicAdd(&A.redo_n[kind], 4);
    at = __shfl_sync(FULL, at, 0);
    if (lane < 4) A.redo[kind * (size_t)A.redo_cap + at + lane] = (item & ~3) | lane;
    return;
  }

  // ------------------------------------------------ reverse
  double qacc = 0.0;    // sum_p w_p Gamma_sp over the face's own cells
  double srcacc = 0.0;  // dL/ddtau(s) from layer 1
  clear();
  __syncwarp();
  bool nz = false;  // whether layer m + 1 has any non-zero M
  for (int m = Llast; m >= 1; --m) {
    const int4 l = layer(m);
    off -= l.z;
    if (m > 1) stage(m - 1, layer(m - 1));
    const bool near = near_bits >> m & 1;
    if (nz || near) {
      const char2* cells = cells_of(m);
      const int base = base_of(m);
      const int gofs = (int)georow_index(m, 0, 0);
      const int naxis = 4 * l.w + 1;
      bool any = false;
      for (int T = 0; T < l.z; T += 32) {
        const int t = T + lane;
        CellIn c;
        fetch_face_cell(Q, c, min(t, l.z - 1), base, cells);
        const int a1 = abs(c.t1), a2 = abs(c.t2);
        const int go = gofs + a1 * (m + 1) + a2;
        double* sc = org + c.t1 * W + c.t2;
        double lam = 0.0, tin = 0.0, tout = 0.0;
        bool rate = false;
        if (near) {
          const double2 tt = stk[off + min(t, l.z - 1)];
          tin = tt.x;
          tout = tt.y;
          rate = bits_of(tin) < a.tab.tau_max_bits;
        }
        if (nz) {
          // users: the cell's own offsets and one step outwards along each axis; from an
          // axis (t = 0, at the front of the table) that is a step to either side
          const int d1 = c.t1 < 0 ? -W : W, d2 = c.t2 < 0 ? -1 : 1;
          double sum = (sc[0] + sc[d1]) + (sc[d2] + sc[d1 + d2]);
          if (T < naxis) sum = axis_users(sc, sum, W, c.t1, c.t2);
          lam = __ldg(&a.kappa[go]) * sum;
        }
        double mup = lam;
        const bool act = t < l.z && in_window(c);
        if (act && (rate || nonzero(lam))) {
          const GeoRow* gr = a.georow + go;
          const double dcell = c.dtp * __ldg(&gr->ds);
          const bool own = (Q.d == 2) || (Q.d == 1 ? a2 < m : (a1 < m && a2 < m));
          int64_t cell = Q.off + c.gidx;
          if (Q.d == 2) {
            const int x1 = wrapc(Q.c1 + c.t1, Q.N), x2 = wrapc(Q.c2 + c.t2, Q.N);
            cell = Q.off + (x1 * Q.N + x2) * Q.N + wrapc(Q.cd + Q.sg * m, Q.N);
          }
          double ndir = 0.0;
          const double wp = own && rate ? __ldg(&A.w[cell]) : 0.0;
          if (nonzero(wp))
            mup = direct_terms(a, Q.nd_thick, Q.nd_thin,
                               __ldg(reinterpret_cast<const double2*>(gr) + 3), &a.invn[cell], wp,
                               c.dtp, dcell, tin, tout, lam, ndir, qacc);
          const double contrib = fma(dcell, lam, ndir);
          if (nonzero(contrib)) atomicAdd(&A.dlogn[cell], contrib);
          any = any || nonzero(mup);
        }
        __syncwarp();  // all reads before any write
        if (act) *sc = mup * __ldg(&a.ikappa[go]);
        __syncwarp();
      }
      nz = __any_sync(FULL, any);
      if (m == 1 && lane < l.z) {  // (kappa = 1 in layer 1; slots outside the window are 0)
        const char2 v = cells[lane];
        srcacc = org[v.x * W + v.y] * (0.5 * __ldg(&a.georow[gofs + abs(v.x) * 2 + abs(v.y)].ds));
      }
    }
    cp_async_wait_all();
    __syncwarp();
  }
  // per-face reductions: dL/dlog Ndot, and the source cell (its own rate, once per
  // source, and its dtau's adjoint)
  double lam_s = 0.0, ndir_s = 0.0;
  if (Q.first && lane == 0) {
    const double tout = Q.half_dts;
    const double ws = A.w[Q.scell];
    if (bits_of(tout) <= bits_of(a.tau_lim)) {
      qacc += ws * (Q.nd * (tab_eval(a.tab.h, a.tab, 0.0) * (0.5 * Q.thin_fac)));
    } else {
      const double fct = Q.nd * Q.inv_cell3 * a.invn[Q.scell];
      const double G = fct * (tab_eval(a.tab.g, a.tab, 0.0) - tab_eval(a.tab.g, a.tab, tout));
      qacc += ws * G;
      lam_s = -ws * fct * tab_slope(a.tab.g, a.tab, tout);
      ndir_s = -ws * G;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    qacc += __shfl_down_sync(FULL, qacc, o);
    srcacc += __shfl_down_sync(FULL, srcacc, o);
  }
  if (lane == 0) {
    if (qacc != 0.0) atomicAdd(&A.dndot[s], qacc);
    const double cs = (2.0 * Q.half_dts) * (srcacc + 0.5 * lam_s) + ndir_s;
    if (cs != 0.0) atomicAdd(&A.dlogn[Q.scell], cs);
  }
}

__global__ void __launch_bounds__(256, 2) k_bwd_faces(BwdArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TraceArgs& a = A.t;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* my = smem_raw + (size_t)wid * rates_warp_bytes(a.hcap, 4);
  double2* stk = A.stack + ((size_t)blockIdx.x * (blockDim.x >> 5) + wid) * A.stack_cap;
  for (;;) {
    int it = 0;
    if (lane == 0) it = a.item_begin + atomicAdd(a.queue, 1);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= a.n_items) break;
    bwd_face(A, a.items[4 * it], lane, my, stk);
    __syncwarp();
  }
}

constexpr int kBwdBlock = 128;
constexpr int kBwdWarps = 8;

static const void* bwd_kernel(int block) {
  return block == 32 ? (const void*)k_trace_faces_bwd_warp<kBwdWarps>
                     : block == 4 ? (const void*)k_bwd_faces : (const void*)k_trace_faces_bwd<kBwdBlock>;
}
static int bwd_threads(int block, int wpb) {
  return block == 32 ? kBwdWarps * 32 : block == 4 ? wpb * 32 : kBwdBlock;
}

// block 32: warp mode (kBwdWarps warps per CTA, one stack per warp); 4: whole faces (wpb
// warps per CTA); 128: CTAs.
cudaError_t launch_trace_bwd(Grid& g, const TraceArgs& t, const BwdLaunch& L, const double* w,
                             double* dlogn, double* dndot_merged, double2* stack) {
  BwdArgs A;
  A.t = t;
  A.w = w;
  A.dlogn = dlogn;
  A.dndot = dndot_merged;
  A.stack = stack;
  A.stack_cap = L.stack_cap;
  A.lcap = L.lcap;
  A.exit = L.exit ? 1 : 0;
  A.redo = L.redo;
  A.redo_n = L.redo_n;
  A.redo_cap = L.redo_cap;
  A.split_src = L.split_src;
  A.n_dev = L.n_dev;
  const void* fn = bwd_kernel(L.block);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.smem);
  if (e != cudaSuccess) return e;
  void* params[] = {&A};
  e = cudaLaunchKernel(fn, dim3(L.grid), dim3(bwd_threads(L.block, L.wpb)), params, L.smem, g.stream);
  count_launch();
  return e;
}

size_t bwd_face_smem_bytes(int hcap) { return rates_warp_bytes(hcap, 4); }

int bwd_max_grid(size_t smem, int block, int wpb) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void* fn = bwd_kernel(block);
  const int threads = bwd_threads(block, wpb);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem);
  if (e != cudaSuccess) return 0;
  return per * sms;
}

// dL/dlog Ndot of each input source from its merged source: Gamma is linear in
// the merged rate, so each member gets its share.
__global__ void k_dndot_inputs(int nsrc, const int* __restrict__ src_of_input,
                               const double* __restrict__ ndot_in,
                               const double* __restrict__ ndot_merged,
                               const double* __restrict__ dmerged, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nsrc) return;
  const int m = src_of_input[i];
  const double nm = ndot_merged[m];
  out[i] = nm > 0.0 ? (ndot_in[i] / nm) * dmerged[m] : 0.0;
}

cudaError_t launch_dndot_inputs(Grid& g, const double* dmerged, double* out) {
  const int T = 256;
  k_dndot_inputs<<<(g.nsrc_in + T - 1) / T, T, 0, g.stream>>>(g.nsrc_in, g.src_of_input,
                                                               g.ndot_in, g.ndot, dmerged, out);
  count_launch();
  return cudaGetLastError();
}

}  // namespace asora
