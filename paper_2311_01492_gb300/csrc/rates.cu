// Batched trace of the photo-ionisation rates (RT_SCHED_BATCHED and its early exit; arXiv
// 2311.01492, Sec. 3.1-3.3), with the geometric weights unless said otherwise.
//
// The work items, their order and the geometry are those of trace.cu: a face of a
// source is a square pyramid whose layer m depends only on layer m - 1, split into
// four quadrants.  An item is traced in two parts.
//
// While a layer has cells with tau_out below the tables' bound 2^E1, the recurrence
// of trace.cu is evaluated as written there, so that every optical depth has the bits
// it has in the other schedules (a rate differs in how its constant factors are
// grouped).  Once every cell of a layer is beyond the bound, every
// later tau_in (a convex combination plus non-negative increments) is too, and every
// later rate is exactly 0: the early exit stops there, the full schedule goes on and
// forms the remaining column densities in the scaled form below.
//
// Scaled form.  The geometric weights of a cell at transverse offsets (a1, a2) of
// layer m are (1 - a1/m | a1/m) times (1 - a2/m | a2/m); with kappa_m(a1, a2) =
// C(m, a1) C(m, a2) (binomial coefficients) and S = kappa tau_out they all become
// one, by Pascal's rule C(m, a) (1 - a/m) = C(m-1, a), C(m, a) a/m = C(m-1, a-1):
//
//   v = kappa tau_in  = S(a1,a2) + S(a1-1,a2) + S(a1,a2-1) + S(a1-1,a2-1)
//   S = kappa tau_out = fma(dtau, kappa ds, v)
//
// (S of layer m - 1 on the right of v; slots outside that layer are zero).  A cell
// costs three additions and one fused multiply-add instead of five multiply-adds,
// reads 8 bytes of geometry (kappa ds) instead of 40, and no weight is rounded.
//
// What binds: GB300 issues one FP64 warp instruction per 68-76 scheduler cycles,
// but integer instructions at full rate beside it (measured: DFMA alone 76.1
// cycles, DFMA with 64 integer instructions 78.3).  Two of the three additions
// therefore run on the integer units, where they also round less: one bracket and
// the final sum are formed as 64-bit integers with nine guard bits and rounded to
// nearest once (<= 0.504 ulp of the sum).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "asora_internal.cuh"
#include "device_util.cuh"
#include "faces.cuh"
#include "scaled_sum.cuh"

namespace asora {

// v of a cell from its four slots of the layer before: one addition on the FP64 unit,
// two on the integer units.
__device__ __forceinline__ double bracket_sum(double c1, double c2, double c3, double c4) {
  return round_sum(c1 + c2, pair_sum(c3, c4));
}

static size_t rates_cta_bytes(int h, int slots) {
  return 2 * rates_buf_bytes(h) + (size_t)slots * row_slot_bytes(h);
}

// Row-table slots of a CTA: this layer's and those staged ahead, or one (the next layer's
// table then waits for the end of the layer) where they do not fit.
static int cta_slots(int h, bool ahead) {
  const int n = ahead ? 3 : 2;
  return rates_cta_bytes(h, n) <= 227 * 1024 ? n : 1;
}

size_t rates_smem_bytes(int hcap, int mode) {
  return mode <= 4 ? rates_warp_bytes(hcap, mode)
                   : rates_cta_bytes(hcap, cta_slots(hcap, mode & kAhead));
}

// The source cell (q = 0), once per source.
__device__ __forceinline__ void source_rate(const TraceArgs& a, const Quad& Q, unsigned& nrate) {
  const bool thin = bits_of(Q.half_dts) <= bits_of(a.tau_lim);
  double dG;
  if (thin)
    dG = Q.nd * (tab_eval(a.tab.h, a.tab, 0.0) * (0.5 * Q.thin_fac));
  else
    dG = Q.nd * ((tab_eval(a.tab.g, a.tab, 0.0) - tab_eval(a.tab.g, a.tab, Q.half_dts)) *
                 Q.inv_cell3);
  ++nrate;
  if (nonzero(dG)) atomicAdd(&(thin ? a.gamma : a.thick)[Q.scell], dG);
}

// The same with optical-depth-modulated weights; r: where s is in the reciprocals.
__device__ __forceinline__ double interp_od(const TraceArgs& a, const Weights& w, const double* s,
                                            const double* r, const int d1, const int d2) {
  return od_interp_r(w.w12.x, w.w12.y, w.w34.x, w.w34.y, s[0], s[-d1], s[-d2], s[-d1 - d2], r[0],
                     r[-d1], r[-d2], r[-d1 - d2], a.neg_zero);
}

// The rate of a cell of layer m >= 1 whose tau_in is within the tables (Eq. sugg; thin
// limit Eq. gammalocal).  The thick terms are summed without their factor 1/n_HI,
// which is the cell's own and is applied once to the sum (k_add_thick): one product
// and one gather less per rate.  FP64 issue binds where rates are everywhere, and an
// instruction that is predicated off takes its turn, so thin and thick cells share theirs
// (a thin one subtracts zero), and which it is comes from the geometry row
// (dtau ds <= tau_lim as a bound on dtau), not from a product.  250^3, 1e5 sources, nearly
// ionised: 190.4 ms with the product, two branches and a comparison of doubles with zero,
// 168.5 in this form.
template <bool FACE>
__device__ __forceinline__ void deposit_rate(const TraceArgs& a, const Quad& Q, const int m,
                                             const CellIn& c, const GeoRow* __restrict__ gr,
                                             const double tin, const double tout,
                                             unsigned& nrate) {
  const int a1 = FACE ? abs(c.t1) : c.t1, a2 = FACE ? abs(c.t2) : c.t2;
  const bool own = ((Q.d == 2) || (Q.d == 1 ? a2 < m : (a1 < m && a2 < m))) &&
                   (FACE || ((a1 > 0 || Q.q1 > 0) && (a2 > 0 || Q.q2 > 0)));
  if (!own) return;
  const double2 gv = __ldg(reinterpret_cast<const double2*>(gr) + 3);  // invv, thin
  int64_t cell = Q.off + c.gidx;
  if (Q.d == 2) {  // gathered from the rotated copy
    const int x1 = wrapc(Q.c1 + Q.q1 * c.t1, Q.N), x2 = wrapc(Q.c2 + Q.q2 * c.t2, Q.N);
    cell = Q.off + (x1 * Q.N + x2) * Q.N + wrapc(Q.cd + Q.sg * m, Q.N);
  }
  const bool thin = bits_of(c.dtp) <= bits_of(__ldg(&gr->lim));
  double* out = thin ? a.gamma : a.thick;
  double dG;
  if (a.tab.kind == RT_TABLE_GREY_EXACT) {
    const double t = thin ? tab_eval(a.tab.h, a.tab, tin)
                          : tab_eval(a.tab.g, a.tab, tin) - tab_eval(a.tab.g, a.tab, tout);
    dG = (thin ? Q.nd_thin : Q.nd_thick) * (t * (thin ? gv.y : gv.x));
  } else {
    const Chord x = tab_chord(thin ? a.tab.h : a.tab.g, a.tab, tin);
    Chord y = {0.0, 0.0, 0.0};
    if (!thin) y = tab_chord(a.tab.g, a.tab, tout);
    const double t = fma(x.c1, x.tau, x.c0) - fma(y.c1, y.tau, y.c0);
    dG = (thin ? Q.nd_thin : Q.nd_thick) * (t * (thin ? gv.y : gv.x));
  }
  ++nrate;
  if (nonzero(dG)) atomicAdd(&out[cell], dG);
}

// Optical depth through a cell that a quadrant owns, to its place in C order.
__device__ __forceinline__ void write_column(const TraceArgs& a, const Quad& Q, const int m,
                                             const CellIn& c, const double tout) {
  const bool own = ((Q.d == 2) || (Q.d == 1 ? c.t2 < m : (c.t1 < m && c.t2 < m))) &&
                   (c.t1 > 0 || Q.q1 > 0) && (c.t2 > 0 || Q.q2 > 0);
  if (!own) return;
  int64_t cell = Q.off + c.gidx;
  if (Q.d == 2) {
    const int x1 = wrapc(Q.c1 + Q.q1 * c.t1, Q.N), x2 = wrapc(Q.c2 + Q.q2 * c.t2, Q.N);
    cell = Q.off + (x1 * Q.N + x2) * Q.N + wrapc(Q.cd + Q.sg * m, Q.N);
  }
  a.coldens[cell] = tout;
}

// Doubles of the part of a layer buffer that an item can read before it writes it
// (the rim of each layer), from the buffer's start.
__device__ __forceinline__ int zero_count(int R2, int h) {
  return (min(h, isqrt_i(R2 >> 1)) + 2) * (h + 2);
}

// tau_out -> S (INV: P = kappa / tau_out) for the cells of layer m (and whatever else
// lies in its square).
template <int GS, bool INV = false>
__device__ __forceinline__ void scale_layer(const TraceArgs& a, double* buf, const int W,
                                            const int m, const int h, const int gt) {
  const int H = min(m, h) + 1;
  const double* __restrict__ k = a.kappa + georow_index(m, 0, 0);
  for (int t = gt; t < H * H; t += GS) {
    const int a1 = t / H, a2 = t - a1 * H;
    double* p = &buf[(a1 + 1) * W + a2 + 1];
    const double kappa = __ldg(&k[a1 * (m + 1) + a2]);
    *p = INV ? quick_div(kappa, *p) : kappa * *p;
  }
}

// The same for a whole face.
template <bool INV>
__device__ __forceinline__ void scale_face(const TraceArgs& a, double* buf, const int W, const int m,
                                           const int h, const int lane) {
  const int H = min(m, h), S = 2 * H + 1;
  const double* __restrict__ k = a.kappa + georow_index(m, 0, 0);
  for (int t = lane; t < S * S; t += 32) {
    const int t1 = t / S - H, t2 = t % S - H;
    double* p = &buf[(t1 + h + 1) * W + t2 + h + 1];
    const double kappa = __ldg(&k[abs(t1) * (m + 1) + abs(t2)]);
    *p = INV ? quick_div(kappa, *p) : kappa * *p;
  }
}

// MODE 1, 2: as many quadrants of one face (from `item` on) by one warp, 32 / MODE
// lanes each with a layer buffer of its own: the quadrants have the same cells, so they
// share the row tables, the geometry loads and the work per layer.  A buffer is updated
// in place, in descending flat order: the slots a cell reads have flat indices not
// above its own, so none is rewritten before it is read.
// MODE 4: a whole face by one warp, for small layers, where the axis lines that two
// quadrants share are a large part (1.25 cells per cell of the ball at R = 15, 1.47 at
// 8).  The cells of a layer come from a table (k_face_tables) in descending order of
// their quadrant position, the images of a position together: the same argument holds.
// The indices and dtau of the next cells (of the next layer at a layer's
// end) are loaded before a step is computed; a step of the scaled part takes two sets
// of 32 cells, whose chains overlap.
//
// OD: optical-depth-modulated weights (od_interp_r).  Each slot's r = 1/max(tau_out,
// tau_w0) lies beside the layer in a global scratch of the warp (rbuf; shared memory for
// both would halve the resident warps, and this part is FP64-bound).  Once all is opaque,
// and beyond tau_w0, every product r tau is one and the normalised sum is the weighted
// harmonic mean: with P = kappa / tau_out,
//   D = kappa / tau_in = P(a1,a2) + P(a1-1,a2) + P(a1,a2-1) + P(a1-1,a2-1)
//   P = kappa / (kappa / D + dtau ds) = D / fma(dtau, D (ds / kappa), 1)
// one division instead of two, and no weights.
template <int MODE, bool EXIT, bool OD>
__device__ __forceinline__ void rates_item_warp(const TraceArgs& a, const int item, const int lane,
                                                unsigned char* __restrict__ sm,
                                                double* __restrict__ rbuf, const int h,
                                                unsigned& nrate) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool FACE = MODE == 4;
  constexpr int K = FACE ? 1 : MODE;
  constexpr int P = 32 / K;  // lanes, and cells of a set, per quadrant (or face)
  const int W = FACE ? 2 * h + 3 : h + 2;
  const int TS = FACE ? face_slot_bytes(h) : row_slot_bytes(h);
  const int lq = lane % P;
  const Quad Q = quad_setup(a, item + lane / P);
  if (lane == 0 && Q.first) source_rate(a, Q, nrate);
  double* buf = reinterpret_cast<double*>(sm + (FACE ? 0 : (lane / P) * rates_buf_bytes(h)));
  unsigned char* tab = sm + (FACE ? face_layer_bytes(h) : K * rates_buf_bytes(h));
  double* const org = FACE ? buf + (h + 1) * (W + 1) : buf + W + 1;  // slot of (0, 0)
  double* const rorg =
      OD ? rbuf + (FACE ? (h + 1) * (W + 1) : (lane / P) * (h + 2) * (h + 2) + W + 1) : nullptr;
  if (FACE) {
    const int hz = min(h, isqrt_i(Q.R2 >> 1));
    for (int t = (h - hz) * W + lane; t < (h + hz + 3) * W; t += 32) buf[t] = 0.0;
    if (lane == 0) buf[0] = 0.0;
  } else {
    for (int t = lq, n = zero_count(Q.R2, h); t < n; t += P) buf[t] = 0.0;
  }
  if (Q.Lmax < 1) return;
  // the row tables serve all K quadrants: those of a window wider by one cell on one
  // side leave cells out (in_window below); the face tables know no window
  const int lim1 = K > 1 ? max(Q.lim1, __shfl_xor_sync(FULL, Q.lim1, P)) : Q.lim1;
  const int lmin1 = K > 1 ? min(Q.lim1, __shfl_xor_sync(FULL, Q.lim1, P)) : Q.lim1;
  const int ent = first_layer_entry(a, Q.R2, FACE ? h : min(lmin1, Q.lim2));
  const int4* __restrict__ lays = FACE ? a.ftab_lay : a.rtab_lay;
  const unsigned char* __restrict__ blobs = FACE ? a.ftab : a.rtab;

  // fetch side: the layer whose cells are being loaded
  int m = 0, sq = 0, kofs = -1, base = 0, T0 = -1;
  // layers m + 1 and m + 2: blob offset, bytes, cells, half-width
  int4 lay = make_int4(0, 0, 0, 0), lay2 = lay;
  const int* rowpre = nullptr;
  const unsigned char* rowof = nullptr;
  const char2* cells = nullptr;
  bool bad = FACE && ent < 0;
  auto stage = [&]() {  // table of layer m + 1
    unsigned char* dst = tab + ((m + 1) & 1) * TS;
    if (FACE || ent >= 0) {
      if (lay.y > TS) bad = true;
      else stage_rows<32>(blobs + lay.x, lay.y, dst, lane);
    } else {
      while (sq * sq > Q.R2 - (m + 1) * (m + 1)) --sq;
      const int H = min(m + 1, sq);
      if (H > h) {
        bad = true;
      } else {
        const int nr = min(H, lim1) + 1;
        int* pre = reinterpret_cast<int*>(dst);
        quad_rows_warp(Q.R2 - (m + 1) * (m + 1), H, nr, Q.lim2, pre,
                       reinterpret_cast<unsigned char*>(pre + nr + 1), lane);
        lay.w = nr - 1;
      }
    }
  };
  auto next_layer = [&]() {  // makes m + 1 the fetched layer (its table has been staged)
    cp_async_wait_all();
    __syncwarp();
    T0 = -1;
    if (bad || m >= Q.Lmax || m >= a.kap_mmax) {
      if ((bad || m < Q.Lmax) && lane == 0) atomicOr(a.err, bad ? ERR_LAYER_CAP : ERR_GEO);
      return;
    }
    ++m;
    kofs += m * m;
    if (FACE) {
      cells = reinterpret_cast<const char2*>(tab + (m & 1) * TS);
      T0 = lay.z - 1;
    } else {
      rowpre = reinterpret_cast<const int*>(tab + (m & 1) * TS);
      rowof = reinterpret_cast<const unsigned char*>(rowpre + lay.w + 2);
      T0 = (ent >= 0 ? lay.z : rowpre[lay.w + 1]) - 1;
    }
    base = wrapc(Q.cd + Q.sg * m, Q.N) * Q.md + Q.org;
    if (m < Q.Lmax) {
      if (FACE || ent >= 0) {
        lay = lay2;
        if (m + 1 < Q.Lmax) lay2 = __ldg(&lays[ent + m + 1]);
      }
      stage();
    }
  };
  auto in_window = [&](const CellIn& c) {
    return (K == 1 && !FACE) || (c.t1 <= Q.lim1 && c.t2 <= Q.lim2);
  };
  auto fetch = [&](CellIn& c, int t) {  // the cell and its offset in the geometry rows
    if (FACE) fetch_face_cell(Q, c, t, base, cells);
    else fetch_cell(Q, c, t, base, rowpre, rowof);
    return kofs + (FACE ? abs(c.t1) : c.t1) * (m + 1) + (FACE ? abs(c.t2) : c.t2);
  };
  // slots one step towards the source along t1 and t2 (faces: the slot itself on an axis)
  auto d1_of = [&](const CellIn& c) { return FACE ? sgn_i(c.t1) * W : W; };
  auto d2_of = [&](const CellIn& c) { return FACE ? sgn_i(c.t2) : 1; };

  sq = isqrt_i(Q.R2 - 1);
  if (ent >= 0) {
    lay = __ldg(&lays[ent]);
    if (Q.Lmax > 1) lay2 = __ldg(&lays[ent + 1]);
  }
  if (!bad) stage();
  next_layer();
  if (T0 < 0) return;
  // ---- cells with rates
  bool opaque = true;  // every cell of this lane in the layer has tau_out beyond the bound
  CellIn nc;
  Weights nw;
  const GeoRow* ng;
  auto prefetch_rated = [&]() {
    ng = a.georow + fetch(nc, max(T0 - lq, 0));
    nw = load_weights(ng);
  };
  prefetch_rated();
  // Layer 1 (one step): from the source's centre to its entry plane.  In quadrants that stop
  // at the opaque layer it is folded into the weights, tau / 2 as the source's slot: half
  // the code, whose fetches count where items are short (128^3, early exit, 5e3 sources of
  // R = 33: 0.47 -> 0.41 ms; longer items lose up to 6%, faces 3%).
  constexpr bool FOLD = EXIT && !OD && !FACE;
  if (FOLD) {
    if (lq == 0) *org = Q.half_dts;
    nw.w12.x *= nw.ds;
    nw.w12.y *= nw.ds;
    nw.w34.x *= nw.ds;
    nw.w34.y *= nw.ds;
    __syncwarp();
  }
  // A layer's last step ends with the test whether all of it is opaque (2^E1 (1 + 2^-40);
  // the margin covers the rounding of later layers).
  auto step = [&](auto first) {
    constexpr bool FIRST = decltype(first)::value;
    const CellIn c = nc;
    const Weights w = nw;
    const GeoRow* gr = ng;
    const int mc = m, Tc = T0;
    const bool last = Tc < P;
    T0 -= P;
    if (last) next_layer();
    if (T0 >= 0) prefetch_rated();
    double* sc = org + c.t1 * W + c.t2;
    double tin;
    if constexpr (FIRST) tin = Q.half_dts * w.ds;  // source centre to the layer's entry plane
    else if constexpr (OD) tin = interp_od(a, w, sc, rorg + c.t1 * W + c.t2, d1_of(c), d2_of(c));
    else tin = interp(a, w, sc, d1_of(c), d2_of(c));
    const double tout = fma(c.dtp, w.ds, tin);
    __syncwarp();  // all reads before any write
    if (Tc - lq >= 0 && in_window(c)) {
      *sc = tout;
      if (OD) rorg[c.t1 * W + c.t2] = od_recip(tout, a.tau_w0);
      opaque = opaque && bits_of(tout) >= a.exit_bits;
      if (bits_of(tin) < a.tab.tau_max_bits)
        deposit_rate<FACE>(a, Q, mc, c, gr, tin, tout, nrate);
    }
    __syncwarp();
    if (!last) return false;
    const bool all = __all_sync(FULL, opaque);
    opaque = true;
    return all;
  };
  // (OD: the scaled form also needs every column beyond tau_w0)
  const bool scalable = !OD || bits_of(a.tau_w0) <= a.exit_bits;
  bool done = !FOLD && step(std::true_type()) && (EXIT || scalable);
  while (T0 >= 0 && !done) done = step(std::false_type()) && (EXIT || scalable);
  if (EXIT || T0 < 0) {
    cp_async_wait_all();  // (a copy may be in flight)
    return;
  }
  // ---- no rates any more: the column densities in scaled form
  if (FACE) scale_face<OD>(a, buf, W, m - 1, h, lane);
  else scale_layer<P, OD>(a, buf, W, m - 1, h, lq);
  __syncwarp();
  const double* __restrict__ geo = OD ? a.dsik : a.kap;
  CellIn ne;
  auto prefetch = [&]() {
    nc.kds = __ldg(&geo[fetch(nc, max(T0 - lq, 0))]);
    if (T0 >= P) ne.kds = __ldg(&geo[fetch(ne, max(T0 - P - lq, 0))]);
  };
  auto column = [&](const CellIn& c, const double* s) {  // S (P) of the cell at slot s
    const int d1 = d1_of(c), d2 = d2_of(c);
    const bool z1 = FACE && c.t1 == 0, z2 = FACE && c.t2 == 0;  // nothing beyond an axis
    const double v = bracket_sum(s[0], z1 ? buf[0] : s[-d1], z2 ? buf[0] : s[-d2],
                                 z1 || z2 ? buf[0] : s[-d1 - d2]);
    return OD ? quick_div(v, fma(c.dtp, v * c.kds, 1.0)) : fma(c.dtp, c.kds, v);
  };
  prefetch();
  while (T0 >= 0) {
    const CellIn c = nc, e = ne;
    const int Tc = T0;
    T0 -= 2 * P;
    if (T0 < 0) next_layer();
    if (T0 >= 0) prefetch();
    double* sc = org + c.t1 * W + c.t2;
    const bool in_c = Tc - lq >= 0 && in_window(c);
    if (Tc >= P) {  // (one block, so that the two chains interleave)
      double* se = org + e.t1 * W + e.t2;
      const double v = column(c, sc);
      const double y = column(e, se);
      __syncwarp();  // all reads before any write
      if (in_c) *sc = v;
      if (Tc - P - lq >= 0 && in_window(e)) *se = y;
    } else {
      const double v = column(c, sc);
      __syncwarp();
      if (in_c) *sc = v;
    }
    __syncwarp();
  }
}

// One quadrant item by a CTA of GS threads: sources too wide for warps, and whatever has
// too few items to fill the GPU.  Two layer buffers and a barrier per layer; the row
// tables are staged one layer ahead.  AHEAD, for launches of few items, where the time
// of a layer is what counts: tables two layers ahead, so that each thread loads the
// indices, dtau and weights of its first cell of the next layer before it computes this
// one (more registers and shared memory than a full GPU has to spare: 128^3, 40 sources
// of R = 40: 0.21 against 0.12 ms).
// WHAT: rates, rates with the early exit, or the column densities of one source (as
// optical depths: launch_tau_to_coldens divides by sigma0 on all SMs).
enum { RATES = 0, RATES_EXIT = 1, COLDENS = 2 };

template <int GS, int WHAT, bool AHEAD>
__device__ __forceinline__ void rates_item_cta(const TraceArgs& a, const int item, const int gt,
                                               unsigned char* __restrict__ sm, const int h,
                                               const int slots, unsigned& nrate) {
  constexpr int D = AHEAD ? 2 : 1;  // layers that the tables are staged ahead (slots == D + 1)
  const int W = h + 2;
  const int TS = row_slot_bytes(h);
  double* cur = reinterpret_cast<double*>(sm);
  double* prev = reinterpret_cast<double*>(sm + rates_buf_bytes(h));
  unsigned char* tab = sm + 2 * rates_buf_bytes(h);
  const int wid = gt >> 5, lane = gt & 31;
  const Quad Q = quad_setup(a, item);
  if (gt == 0 && Q.first) {
    if (WHAT == COLDENS) a.coldens[Q.scell] = Q.half_dts;
    else source_rate(a, Q, nrate);
  }
  for (int t = gt, n = zero_count(Q.R2, h); t < n; t += GS) cur[t] = prev[t] = 0.0;
  if (Q.Lmax < 1) return;
  // tables know no window: cells outside it are left out one by one
  const int ent = first_layer_entry(a, Q.R2, h);
  int sq = isqrt_i(Q.R2 - 1);
  auto half_width = [&](int m) {  // for m ascending
    while (sq * sq > Q.R2 - m * m) --sq;
    return min(m, sq);
  };
  bool bad = false;
  auto stage = [&](int m, int H) {  // row table of layer m (waited for separately)
    unsigned char* dst = tab + (slots > 1 ? m % (D + 1) * TS : 0);
    if (H > h) {
      bad = true;
    } else if (ent >= 0) {
      const int4 lay = __ldg(&a.rtab_lay[ent + m - 1]);
      stage_rows<GS>(a.rtab + lay.x, lay.y, dst, gt);
    } else if (wid == 0) {
      int* pre = reinterpret_cast<int*>(dst);
      quad_rows_warp(Q.R2 - m * m, H, H + 1, h, pre,
                     reinterpret_cast<unsigned char*>(pre + H + 2), lane);
    }
  };
  struct Layer {
    const int* rowpre;
    const unsigned char* rowof;
    int total, base, gofs;
  };
  auto layer = [&](int m, int H) {
    Layer L;
    L.rowpre = reinterpret_cast<const int*>(tab + (slots > 1 ? m % (D + 1) * TS : 0));
    L.rowof = reinterpret_cast<const unsigned char*>(L.rowpre + H + 2);
    L.total = L.rowpre[H + 1];
    L.base = wrapc(Q.cd + Q.sg * m, Q.N) * Q.md + Q.org;
    L.gofs = (int)georow_index(m, 0, 0);
    return L;
  };
  struct Ahead {  // a cell and its weights (scaled part: kappa ds in c.kds)
    CellIn c;
    Weights w;
    const GeoRow* gr;
  };
  auto load = [&](Ahead& x, const Layer& L, int m, int t, bool scaled) {
    fetch_cell(Q, x.c, t, L.base, L.rowpre, L.rowof);
    const int o = L.gofs + x.c.t1 * (m + 1) + x.c.t2;
    x.gr = a.georow + o;
    if (scaled) x.c.kds = __ldg(&a.kap[o]);
    else x.w = load_weights(x.gr);
  };
  bool opaque = true;  // every cell of this thread in the layer has tau_out beyond the bound
  auto rated = [&](const Ahead& x, int m, double tin) {  // the cell's column, and its rate
    const double tout = fma(x.c.dtp, x.w.ds, tin);
    if (x.c.t1 > Q.lim1 || x.c.t2 > Q.lim2) return;
    cur[(x.c.t1 + 1) * W + x.c.t2 + 1] = tout;
    if (WHAT == COLDENS) {
      write_column(a, Q, m, x.c, tout);
      return;
    }
    opaque = opaque && bits_of(tout) >= a.exit_bits;
    if (bits_of(tin) < a.tab.tau_max_bits)
      deposit_rate<false>(a, Q, m, x.c, x.gr, tin, tout, nrate);
  };
  int Hc = half_width(1), Hn = 0;  // of this layer and the next
  stage(1, Hc);
  if (Q.Lmax > 1) {
    Hn = half_width(2);
    if (AHEAD && slots > 1) stage(2, Hn);
  }
  cp_async_wait_all();
  group_sync<GS>();
  bool scaled = false, ahead_scaled = false;
  Ahead nx;
  for (int m = 1; m <= Q.Lmax; ++m) {
    if (bad || m > a.kap_mmax) {  // (a layer found too wide when it was to be staged)
      if (gt == 0) atomicOr(a.err, bad ? ERR_LAYER_CAP : ERR_GEO);
      break;
    }
    const Layer L = layer(m, Hc);
    int Hnn = 0;
    if (m + 2 <= Q.Lmax) Hnn = half_width(m + 2);
    if (slots > 1 && m + D <= Q.Lmax) stage(m + D, AHEAD ? Hnn : Hn);
    Ahead x = nx;
    const bool have = AHEAD && slots > 1 && m > 1;  // x: this thread's first cell
    bool x_scaled = ahead_scaled;
    if (AHEAD && slots > 1 && m < Q.Lmax && Hn <= h) {
      const Layer Ln = layer(m + 1, Hn);
      if (gt < Ln.total) load(nx, Ln, m + 1, gt, scaled);
      ahead_scaled = scaled;
    }
    opaque = true;
    if (m == 1) {  // the column from the source centre to the layer's entry plane
      if (gt < L.total) {
        load(x, L, m, gt, false);
        rated(x, m, Q.half_dts * x.w.ds);
      }
    } else {
      for (int t = gt; t < L.total; t += GS) {
        if (t > gt || !have) {
          load(x, L, m, t, scaled);
          x_scaled = scaled;
        }
        const double* s = prev + (x.c.t1 + 1) * W + x.c.t2 + 1;
        if (scaled) {
          if (AHEAD && !x_scaled) x.c.kds = __ldg(&a.kap[x.gr - a.georow]);  // (loaded for a rated layer)
          const double v = fma(x.c.dtp, x.c.kds, bracket_sum(s[0], s[-W], s[-1], s[-W - 1]));
          if (x.c.t1 <= Q.lim1 && x.c.t2 <= Q.lim2) cur[(x.c.t1 + 1) * W + x.c.t2 + 1] = v;
        } else {
          rated(x, m, interp(a, x.w, s, W, 1));
        }
      }
    }
    if (slots == 1 && m < Q.Lmax) {
      group_sync<GS>();  // this layer's table is no longer read
      stage(m + 1, Hn);
    }
    cp_async_wait_all();
    if (WHAT == COLDENS || scaled) {
      __syncthreads();
    } else if (__syncthreads_and(opaque)) {  // as in rates_item_warp
      if (WHAT == RATES_EXIT) break;
      scaled = true;
      scale_layer<GS>(a, cur, W, m, h, gt);
      __syncthreads();
    }
    double* tmp = prev;
    prev = cur;
    cur = tmp;
    Hc = Hn;
    Hn = Hnn;
  }
  cp_async_wait_all();
}

__device__ __forceinline__ void flush_rates(const TraceArgs& a, unsigned nrate) {
  if (!a.rate_cells) return;
  for (int o = 16; o > 0; o >>= 1) nrate += __shfl_down_sync(0xffffffffu, nrate, o);
  if ((threadIdx.x & 31) == 0 && nrate) atomicAdd(a.rate_cells, (unsigned long long)nrate);
}

// Threads per SM that the registers are cut for: 896 (72 registers) where all layers are
// traced: 64 spill (250^3, 200 sources of R = 5..50: 0.323 / 0.260 ms; 128^3, 400: 0.395 /
// 0.335), 80 leave too few CTAs (64^3, 256: 0.202 / 0.198 / 0.215); 1024 with the early
// exit (128^3, 400: 0.067 / 0.071).
constexpr int cta_threads(int what, bool ahead) {
  return ahead ? 512 : what == RATES_EXIT ? 1024 : 896;
}

template <int BLOCK, int WHAT, bool AHEAD>
__global__ void __launch_bounds__(BLOCK, cta_threads(WHAT, AHEAD) / BLOCK)
k_rates_cta(TraceArgs a, int slots) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_item;
  if (a.skip && *a.skip) return;
  unsigned nrate = 0;
  if (AHEAD) {  // as many CTAs as there are items
    const int item = WHAT == COLDENS ? (*a.one_src << 5) | (int)blockIdx.x
                                     : a.items[a.item_begin + blockIdx.x];
    rates_item_cta<BLOCK, WHAT, AHEAD>(a, item, threadIdx.x, smem_raw, a.hcap, slots, nrate);
  } else {
    for (;;) {
      __syncthreads();
      if (threadIdx.x == 0) s_item = a.item_begin + atomicAdd(a.queue, 1);
      __syncthreads();
      const int it = s_item;
      if (it >= a.n_items) break;
      rates_item_cta<BLOCK, WHAT, AHEAD>(a, a.items[it], threadIdx.x, smem_raw, a.hcap, slots,
                                         nrate);
    }
  }
  if (WHAT != COLDENS) flush_rates(a, nrate);
}

// Doubles of one layer buffer of a warp (all its quadrants, or its face).
__host__ __device__ inline size_t warp_slots(int h, int mode) {
  return mode == 4 ? (size_t)(2 * h + 3) * (2 * h + 3) : (size_t)mode * (h + 2) * (h + 2);
}

// Threads of a CTA and CTAs per SM that the registers are cut for.  The scaled part waits
// for loads and shared memory, so warps count: with up to 16 (127 registers), 20 (96) or 24
// (80) per SM a batched trace of 128^3 takes, in one quadrant per warp (half-width 23, 5e3
// sources) 4.76 / 4.41 / 4.28 ms, in whole faces (11, 2e4) 3.02 / 2.76 / 2.65, in two
// quadrants (19, 8e3; 80 registers spill) 4.28 / 4.02 / 4.82.  With optical-depth weights
// 7.19 / 7.26 / 7.31, with rates everywhere 2.33 / 2.29 / 2.31: FP64-bound.
__host__ __device__ constexpr int rates_warps(int mode, bool exit, bool od) {
  return od ? 8 : mode == 2 || (mode == 4 && exit) ? 4 : 3;
}
__host__ __device__ constexpr int rates_ctas(int mode, bool exit, bool od) {
  return od ? 2 : mode == 2 || (mode == 4 && exit) ? 5 : 7;
}

template <int MODE, bool EXIT, bool OD>
__global__ void __launch_bounds__(32 * rates_warps(MODE, EXIT, OD), rates_ctas(MODE, EXIT, OD))
k_rates_warp(TraceArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (a.skip && *a.skip) return;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* my = smem_raw + (size_t)wid * rates_warp_bytes(a.hcap, MODE);
  double* rbuf = nullptr;
  if (OD) {  // finite values in every slot that a zero weight may read
    const size_t n = warp_slots(a.hcap, MODE);
    rbuf = a.scratch + ((size_t)blockIdx.x * (blockDim.x >> 5) + wid) * n;
    for (size_t t = lane; t < n; t += 32) rbuf[t] = 0.0;
    __syncwarp();
  }
  unsigned nrate = 0;
  for (;;) {
    int it = 0;
    if (lane == 0) it = a.item_begin + atomicAdd(a.queue, 1);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= a.n_items) break;
    rates_item_warp<MODE, EXIT, OD>(a, a.items[it * MODE], lane, my, rbuf, a.hcap, nrate);
    __syncwarp();
  }
  flush_rates(a, nrate);
}

// mode: quadrants per warp (1, 2), 4: a whole face per warp, or threads of a CTA (128,
// 256; with kAhead 128, 256, 512)
static const void* rates_kernel(int mode, int what, bool od) {
  const bool exit = what == RATES_EXIT;
#define ASORA_WARP(M)                                                                          \
  (od ? exit ? (const void*)k_rates_warp<M, true, true> : (const void*)k_rates_warp<M, false, true> \
      : exit ? (const void*)k_rates_warp<M, true, false>                                       \
             : (const void*)k_rates_warp<M, false, false>)
#define ASORA_CTA(B, AHEAD)                                      \
  (od ? nullptr : exit ? (const void*)k_rates_cta<B, RATES_EXIT, AHEAD> \
                       : (const void*)k_rates_cta<B, RATES, AHEAD>)
#define ASORA_AHEAD(B) \
  (what == COLDENS ? (const void*)k_rates_cta<B, COLDENS, true> : ASORA_CTA(B, true))
  switch (mode) {
    case 1: return ASORA_WARP(1);
    case 2:
      return od ? nullptr : exit ? (const void*)k_rates_warp<2, true, false>
                                 : (const void*)k_rates_warp<2, false, false>;
    case 4: return ASORA_WARP(4);
    case 128: return ASORA_CTA(128, false);
    case 256: return ASORA_CTA(256, false);
    case 128 | kAhead: return ASORA_AHEAD(128);
    case 256 | kAhead: return ASORA_AHEAD(256);
    case 512 | kAhead: return ASORA_AHEAD(512);
    default: return nullptr;
  }
#undef ASORA_AHEAD
#undef ASORA_CTA
#undef ASORA_WARP
}

cudaError_t launch_rates(Grid& g, const TraceArgs& a, int mode, int grid, size_t smem, int wpb) {
  const void* fn =
      rates_kernel(mode, a.coldens ? COLDENS : a.early_exit ? RATES_EXIT : RATES,
                   !a.coldens && a.interp_mode == RT_INTERP_OPTICAL_DEPTH);
  if (!fn) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  TraceArgs arg = a;
  int slots = cta_slots(a.hcap, mode & kAhead);
  void* params[] = {&arg, &slots};  // (the warp kernels take the first only)
  e = cudaLaunchKernel(fn, dim3(grid), dim3(mode <= 4 ? wpb * 32 : mode & ~kAhead), params, smem, g.stream);
  count_launch();
  return e;
}

int rates_max_warps(int mode, bool exit, bool od) { return rates_warps(mode, exit, od); }

int rates_max_grid(int mode, size_t smem, int wpb, bool exit, bool od) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void* fn = rates_kernel(mode, exit ? RATES_EXIT : RATES, od);
  if (!fn) return 0;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, mode <= 4 ? wpb * 32 : mode & ~kAhead,
                                                      smem);
  if (e != cudaSuccess) return 0;
  return per * sms;
}

}  // namespace asora
