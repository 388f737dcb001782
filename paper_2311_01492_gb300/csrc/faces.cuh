// What the kernels that trace quadrants or whole faces share (rates.cu, adjoint.cu):
// shared-memory layouts, an item's geometry, cells and their weights.
#pragma once

#include "asora_internal.cuh"
#include "device_util.cuh"

namespace asora {

// ------------------------------------------------------------ shared memory
// Layer buffer: slot of (a1, a2), a1, a2 = -1..h, at (a1+1) W + a2+1, W = h+2 (row
// and column -1 stay zero).  One buffer per warp (updated in place), two per CTA;
// then `slots` row-table slots (device_util.cuh).
__host__ __device__ inline size_t rates_buf_bytes(int h) {
  return ((size_t)(h + 2) * (h + 2) * sizeof(double) + 15) & ~(size_t)15;
}
// Whole faces (mode 4): slot of the signed offsets (t1, t2) at (t1+h+1) W + t2+h+1, W =
// 2h+3, slot 0 always zero; then two slots for the face tables (k_face_tables).
__host__ __device__ inline size_t face_layer_bytes(int h) {
  return ((size_t)(2 * h + 3) * (2 * h + 3) * sizeof(double) + 15) & ~(size_t)15;
}
__host__ __device__ inline int face_slot_bytes(int h) {
  return (2 * (2 * h + 1) * (2 * h + 1) + 15) & ~15;
}
__host__ __device__ inline size_t rates_warp_bytes(int h, int mode) {
  return mode == 4 ? face_layer_bytes(h) + 2 * (size_t)face_slot_bytes(h)
                   : mode * rates_buf_bytes(h) + 2 * (size_t)row_slot_bytes(h);
}
// ----------------------------------------------------------------- quadrants
// One quadrant of a face as a lane sees it: the geometry of trace_face_item
// (trace.cu) and its source's constants.
struct Quad {
  int N, R2, d, sg, q1, q2, lim1, lim2, Lmax;
  int c1, c2, cd;          // source coordinates along t1, t2 and the face's axis
  int md, st1;             // strides of the layer axis and (signed) of a1
  int w1, w2, C1, C2;      // from a1 = w1 (a2 = w2) on, the offset is corrected by C1 (C2)
  int org;                 // offset of (c1, c2) within a layer
  int64_t off, scell;      // first cell of the box, the source's cell
  double half_dts, nd, inv_cell3, thin_fac, nd_thick, nd_thin;
  bool first;              // the one item of a source that has its own cell
  const double* fld;       // dtau, rotated for the z faces: the stride of a2 is 1
};

__device__ __forceinline__ Quad quad_setup(const TraceArgs& a, const int item) {
  Quad Q;
  const int s = item >> 5, f = (item >> 2) & 7, quad = item & 3;
  const SrcDev S = a.src[s];
  const BoxDev B = a.boxes[S.box];
  Q.nd = a.ndot[s];
  Q.N = B.n;
  Q.R2 = a.r2lim[s];
  Q.d = f >> 1;
  Q.sg = (f & 1) ? -1 : 1;
  Q.q1 = (quad & 1) ? -1 : 1;
  Q.q2 = (quad & 2) ? -1 : 1;
  Q.lim1 = Q.q1 > 0 ? B.whi : -B.wlo;
  Q.lim2 = Q.q2 > 0 ? B.whi : -B.wlo;
  Q.Lmax = min(Q.sg > 0 ? B.whi : -B.wlo, isqrt_i(Q.R2));
  Q.off = B.off;
  Q.scell = B.off + ((int64_t)S.i * Q.N + S.j) * Q.N + S.k;
  Q.half_dts = 0.5 * a.dtau[Q.scell];
  Q.inv_cell3 = B.inv_cell3;
  Q.thin_fac = B.thin_fac;
  Q.nd_thick = Q.nd * B.inv_cell3;
  Q.nd_thin = Q.nd * B.thin_fac;
  Q.first = f == 4 && quad == 0;
  const int NN = Q.N * Q.N;
  Q.c1 = Q.d == 0 ? S.j : S.i;
  Q.c2 = Q.d == 2 ? S.j : S.k;
  Q.cd = Q.d == 0 ? S.i : (Q.d == 1 ? S.j : S.k);
  const int m1 = Q.d == 1 ? NN : Q.N;
  Q.md = Q.d == 1 ? Q.N : NN;
  Q.fld = (Q.d == 2 ? a.dtauT : a.dtau) + B.off;
  Q.st1 = Q.q1 * m1;
  Q.w1 = Q.q1 > 0 ? Q.N - Q.c1 : Q.c1 + 1;
  Q.w2 = Q.q2 > 0 ? Q.N - Q.c2 : Q.c2 + 1;
  Q.C1 = -Q.q1 * Q.N * m1;
  Q.C2 = -Q.q2 * Q.N;
  Q.org = Q.c1 * m1 + Q.c2;
  return Q;
}

// First layer entry (rtab_lay) of the item's R^2 limit, or -1 if a window of half-width
// lim clips a layer (or there are no tables).
__device__ __forceinline__ int first_layer_entry(const TraceArgs& a, const int R2, const int lim) {
  if (R2 > a.rtab_max_r2) return -1;
  const int sl = a.rtab_slot[R2];
  return sl >= 0 && a.rtab_hcap[sl] <= lim ? a.rtab_first[sl] : -1;
}

// One cell in flight: transverse offsets along the item's signs (quadrants: >= 0) or
// signed (faces).
struct CellIn {
  int t1, t2, gidx;
  double dtp, kds;
};

__device__ __forceinline__ void fetch_cell(const Quad& Q, CellIn& c, const int t, const int base,
                                           const int* __restrict__ rowpre,
                                           const unsigned char* __restrict__ rowof) {
  c.t1 = rowof[t];
  c.t2 = t - rowpre[c.t1];
  c.gidx = base + c.t1 * Q.st1 + Q.q2 * c.t2 + (c.t1 >= Q.w1 ? Q.C1 : 0) + (c.t2 >= Q.w2 ? Q.C2 : 0);
  c.dtp = __ldg(&Q.fld[c.gidx]);
}

// The same from a face table; a face wraps on either side.
__device__ __forceinline__ void fetch_face_cell(const Quad& Q, CellIn& c, const int t,
                                                const int base, const char2* __restrict__ cells) {
  const char2 v = cells[t];
  c.t1 = v.x;
  c.t2 = v.y;
  const int x1 = Q.c1 + c.t1, x2 = Q.c2 + c.t2;
  c.gidx = base + c.t1 * Q.st1 + c.t2 + (x1 < 0 ? -Q.C1 : x1 >= Q.N ? Q.C1 : 0) +
           (x2 < 0 ? -Q.C2 : x2 >= Q.N ? Q.C2 : 0);
  c.dtp = __ldg(&Q.fld[c.gidx]);
}

// Weights and path length of a cell.
struct Weights {
  double2 w12, w34;
  double ds;
};
__device__ __forceinline__ Weights load_weights(const GeoRow* __restrict__ gr) {
  return {__ldg(reinterpret_cast<const double2*>(gr)),
          __ldg(reinterpret_cast<const double2*>(gr) + 1), __ldg(&gr->ds)};
}

// tau_in of a cell from the interpolants at slot s and up to d1 and d2 before it
// (trace.cu; the slots that a zero weight reads hold a finite value).
__device__ __forceinline__ double interp(const TraceArgs& a, const Weights& w, const double* s,
                                         const int d1, const int d2) {
  return fma(w.w34.y, s[-d1 - d2],
             fma(w.w34.x, s[-d2], fma(w.w12.y, s[-d1], fma(w.w12.x, s[0], a.neg_zero))));
}

}  // namespace asora
