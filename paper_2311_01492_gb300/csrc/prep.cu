// Per-call preparation kernels: field validation, per-cell optical depth
// (Sec. 3.1: dtau = sigma0 * alpha * n_HI), its axis-rotated copy for the
// z faces, 1/n_HI, the source-independent geometry table and source ingest
// (merging of co-located sources, Sec. 3, and longest-first ordering).
#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <type_traits>

#include "asora_internal.cuh"
#include "device_util.cuh"

namespace asora {

// ----------------------------------------------------------- validation
// (writes its own error word, so that it never clears the bits the trace kernels latch)
// All values in [+0, top], by their bits: negative values, -0 and NaN have larger ones.  A
// comparison of doubles takes an FP64 turn: three of them 66 us at 250^3, this 24 (18 by
// its bytes).
__global__ void k_validate_field(const double* __restrict__ v, double top, int64_t ncell,
                                 int* __restrict__ err) {
  bool bad = false;
#pragma unroll 4
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell;
       c += (int64_t)gridDim.x * blockDim.x)
    bad |= bits_of(v[c]) > bits_of(top);
  if (bad) *err = ERR_INPUT;  // (pinned host memory: nothing to clear or to copy back)
}

cudaError_t launch_validate_field(Grid& g, const double* v, double top) {
  k_validate_field<<<1024, 256, 0, g.stream>>>(v, top, g.ncell, g.pin);
  count_launch();
  return cudaGetLastError();
}

// --------------------------------------------------------- per-cell fields
// One 32x32 tile of the (n^2 rows (i,j)) x (n cols k) matrix of a box:
// dtau = ((sigma0*cell)*n_H)*x_HI, invn = 1/(n_H*x_HI), and the transposed
// copy dtauT[k][i][j] so that the z faces read rows of constant k contiguously.
// n_H is the proper density: the given (comoving) one times inv_a3 = a^-3 in an
// expanding background (inv_a3 = 1 otherwise, an exact no-op); cell (in the
// box records) is the proper cell size.  WHAT: 1/n_HI only where it is read; the batched
// rates divide their summed thick terms by n_HI once per cell (k_add_thick) and take
// zeros to sum into, column densities need neither (an FP64 division per cell made this
// kernel 2.4 times its memory time at 250^3).  The call's output field is zeroed here
// too: one launch less.
template <int WHAT>
__global__ void k_precompute(const BoxDev* __restrict__ boxes, const double* __restrict__ nH,
                             const double* __restrict__ xHI, double inv_a3,
                             double* __restrict__ dtau, double* __restrict__ dtauT,
                             double* __restrict__ invn, double* __restrict__ out,
                             const int* __restrict__ skip) {
  __shared__ double tile[32][33];
  if (skip && *skip) return;
  const BoxDev B = boxes[blockIdx.z];
  const int n = B.n;
  const int64_t rows = (int64_t)n * n;
  const int c0 = blockIdx.x * 32;
  if (c0 >= n) return;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int64_t r0 = (int64_t)blockIdx.y * 32; r0 < rows; r0 += (int64_t)gridDim.y * 32) {
    for (int yy = ty; yy < 32; yy += 8) {
      const int64_t r = r0 + yy;
      const int c = c0 + tx;
      if (r < rows && c < n) {
        const int64_t idx = B.off + r * n + c;
        const double nh = nH[idx] * inv_a3, x = xHI[idx];
        const double d = (B.sig_cell * nh) * x;
        dtau[idx] = d;
        if (WHAT == PRE_INVN) invn[idx] = quick_recip(nh * x);
        if (WHAT == PRE_THICK) invn[idx] = 0.0;
        if (out) out[idx] = 0.0;
        tile[yy][tx] = d;
      }
    }
    __syncthreads();
    for (int yy = ty; yy < 32; yy += 8) {
      const int c = c0 + yy;        // k
      const int64_t r = r0 + tx;    // (i,j)
      if (r < rows && c < n) dtauT[B.off + (int64_t)c * rows + r] = tile[tx][yy];
    }
    __syncthreads();
  }
}

cudaError_t launch_precompute(Grid& g, int what, double* out, const int* skip) {
  const int n = g.nmax;
  dim3 grid((n + 31) / 32, (unsigned)std::min<int64_t>(((int64_t)n * n + 31) / 32, 65535), g.nbox);
  auto* k = what == PRE_INVN ? k_precompute<PRE_INVN>
                             : what == PRE_THICK ? k_precompute<PRE_THICK> : k_precompute<PRE_DTAU>;
  k<<<grid, dim3(32, 8), 0, g.stream>>>(g.boxes_d, g.nH, g.xHI, g.inv_a3, g.dtau, g.dtauT, g.invn,
                                        out, skip);
  count_launch();
  return cudaGetLastError();
}

// Optical depths to column densities (division: the quotient is rounded once), for the
// traced part only.
__global__ void k_tau_to_coldens(int64_t n, double sigma0, double* __restrict__ c) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const double v = c[t];
    if (bits_of(v)) c[t] = exact_div(v, sigma0);
  }
}

cudaError_t launch_tau_to_coldens(Grid& g, double* coldens) {
  const int grid = (int)std::min<int64_t>((g.ncell + 255) / 256, 152 * 16);
  k_tau_to_coldens<<<grid, 256, 0, g.stream>>>(g.ncell, g.p.sigma0_cm2, coldens);
  count_launch();
  return cudaGetLastError();
}

// gamma += thick / n_HI (Eq. sugg's 1/n_HI, taken out of the sum over sources).  FP64 issue
// binds while a cell takes more than three instructions (4 fields through memory: 74 us at
// 250^3): 165 us, and 350 with a / b, 1/a^3 always applied and a test in FP64.
template <bool SCALED>
__global__ void k_add_thick(int64_t n, const double* __restrict__ nH, const double* __restrict__ xHI,
                            double inv_a3, const double* __restrict__ thick,
                            double* __restrict__ gamma, const int* __restrict__ skip) {
  if (skip && *skip) return;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n;
       c += (int64_t)gridDim.x * blockDim.x) {
    const double t = thick[c];
    if (bits_of(t)) gamma[c] += quick_div(t, (SCALED ? nH[c] * inv_a3 : nH[c]) * xHI[c]);
  }
}

cudaError_t launch_add_thick(Grid& g, double* gamma, const int* skip) {
  const int grid = (int)std::min<int64_t>((g.ncell + 255) / 256, 152 * 16);
  auto* k = g.inv_a3 != 1.0 ? k_add_thick<true> : k_add_thick<false>;
  k<<<grid, 256, 0, g.stream>>>(g.ncell, g.nH, g.xHI, g.inv_a3, g.invn, gamma, skip);
  count_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------------- geometry
// Entry (m, lo, hi): bilinear weights of Sec. 3.1 for a = lo/m, b = hi/m and
// the path length ds = sqrt(1 + (lo^2+hi^2)/m^2).  Both are computed with
// correctly rounded IEEE division and square root.
// Binomial coefficients C(m, a), a <= m <= kKapMax, at m (m + 1) / 2 + a as the sum
// of two doubles: they grow to 2^(2m), and the products of two are rounded only once
// when they enter kappa and kappa ds.  C(m, a) = C(m, a-1) (m - a + 1) / a.
__global__ void k_binomials(double2* __restrict__ b, int mmax) {
  const int m = blockIdx.x;
  if (m > mmax) return;
  for (int a = threadIdx.x; a <= m; a += blockDim.x) {
    double hi = 1.0, lo = 0.0;
    const int k = min(a, m - a);
    for (int i = 1; i <= k; ++i) {
      const double x = (double)(m - i + 1), y = (double)i;
      double ph = hi * x;
      double pl = fma(hi, x, -ph) + lo * x;
      const double q = (ph + pl) / y;
      const double r = fma(-q, y, ph) + pl;
      const double q2 = r / y;
      hi = q + q2;
      lo = q2 - (hi - q);
    }
    b[m * (m + 1) / 2 + a] = make_double2(hi, lo);
  }
}

// kappa = C(m, a1) C(m, a2) as the sum of two doubles
__device__ __forceinline__ double2 kappa_dd(const double2* __restrict__ b, int m, int a1, int a2) {
  const double2 x = b[m * (m + 1) / 2 + a1], y = b[m * (m + 1) / 2 + a2];
  const double ph = x.x * y.x;
  const double pl = fma(x.x, y.x, -ph) + (x.x * y.y + x.y * y.x);
  const double hi = ph + pl;
  return make_double2(hi, pl - (hi - ph));
}

__global__ void k_geometry(GeoEntry* __restrict__ geo, int mmax) {
  const int m = blockIdx.x + 1;
  if (m > mmax) return;
  const int cnt = (m + 1) * (m + 2) / 2;
  for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
    int hi = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    while (hi * (hi + 1) / 2 > t) --hi;
    while ((hi + 1) * (hi + 2) / 2 <= t) ++hi;
    const int lo = t - hi * (hi + 1) / 2;
    const double x = (double)lo / (double)m;
    const double y = (double)hi / (double)m;
    GeoEntry e;
    e.w1 = (1.0 - x) * (1.0 - y);
    e.wa = x * (1.0 - y);
    e.wb = (1.0 - x) * y;
    e.w4 = x * y;
    e.ds = sqrt(1.0 + (double)(lo * lo + hi * hi) / (double)(m * m));
    const double r2 = (double)(m * m + lo * lo + hi * hi);
    const double fourpi = 12.566370614359172;
    e.invv = 1.0 / (fourpi * r2 * e.ds);
    e.thin = 1.0 / (fourpi * r2);
    e.pad = 0.0;
    geo[geo_index(m, lo, hi)] = e;
  }
}

// Row-major entry (m, a1, a2) with the same correctly rounded expressions.
__global__ void k_geometry_rows(GeoRow* __restrict__ geo, double* __restrict__ kap,
                                double* __restrict__ kappa, double* __restrict__ ikappa,
                                double* __restrict__ dsik, const double2* __restrict__ binom, double tau_lim,
                                int mmax) {
  const int m = blockIdx.x + 1;
  if (m > mmax) return;
  const int cnt = (m + 1) * (m + 1);
  for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
    const int a1 = t / (m + 1), a2 = t - a1 * (m + 1);
    const double x = (double)a1 / (double)m;
    const double y = (double)a2 / (double)m;
    GeoRow e;
    e.w1 = (1.0 - x) * (1.0 - y);
    e.w2 = x * (1.0 - y);
    e.w3 = (1.0 - x) * y;
    e.w4 = x * y;
    e.ds = sqrt(1.0 + (double)(a1 * a1 + a2 * a2) / (double)(m * m));
    e.lim = tau_lim / e.ds;  // the bound itself is a step or two away at most
    for (int k = 0; k < 4 && e.lim * e.ds > tau_lim; ++k)
      e.lim = __longlong_as_double(__double_as_longlong(e.lim) - 1);
    for (int k = 0; k < 4; ++k) {
      const double up = __longlong_as_double(__double_as_longlong(e.lim) + 1);
      if (up * e.ds <= tau_lim) e.lim = up;
    }
    const double r2 = (double)(m * m + a1 * a1 + a2 * a2);
    const double fourpi = 12.566370614359172;
    e.invv = 1.0 / (fourpi * r2 * e.ds);
    e.thin = 1.0 / (fourpi * r2);
    geo[georow_index(m, a1, a2)] = e;
    if (m <= kKapMax) {
      const double2 k = kappa_dd(binom, m, a1, a2);
      kap[georow_index(m, a1, a2)] = fma(k.x, e.ds, k.y * e.ds);
      kappa[georow_index(m, a1, a2)] = k.x;
      const double q = 1.0 / k.x;  // 1/kappa: one Newton step on the two-part kappa
      const double ik = q + q * (fma(-q, k.x, 1.0) - q * k.y);
      ikappa[georow_index(m, a1, a2)] = ik;
      dsik[georow_index(m, a1, a2)] = e.ds * ik;
    }
  }
}

// k = min(mmax, kKapMax): kap holds georow_count(k) values of kappa ds, then as many of
// kappa, 1/kappa and ds/kappa, then scratch: the binomials
cudaError_t launch_geometry(GeoEntry* geo, GeoRow* georow, double* kap, double tau_lim, int mmax,
                            cudaStream_t s) {
  if (mmax < 1) return cudaSuccess;
  double2* binom = reinterpret_cast<double2*>(kap + 4 * georow_count(std::min(mmax, kKapMax)));
  k_binomials<<<std::min(mmax, kKapMax) + 1, 64, 0, s>>>(binom, std::min(mmax, kKapMax));
  count_launch();
  const int64_t nk = georow_count(std::min(mmax, kKapMax));
  k_geometry_rows<<<mmax, 256, 0, s>>>(georow, kap, kap + nk, kap + 2 * nk, kap + 3 * nk, binom,
                                         tau_lim, mmax);
  count_launch();
  k_geometry<<<mmax, 256, 0, s>>>(geo, mmax);
  count_launch();
  return cudaGetLastError();
}

// --------------------------------------------------------- source ingest
__global__ void k_src_keys(const BoxDev* __restrict__ boxes, int nbox, int nsrc,
                           const int32_t* __restrict__ pos, const int32_t* __restrict__ box,
                           const double* __restrict__ ndot, const double* __restrict__ radius,
                           uint64_t* __restrict__ keys, int* __restrict__ idx,
                           int* __restrict__ r2out, int* __restrict__ err) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsrc) return;
  const int b = box ? box[s] : 0;
  bool bad = b < 0 || b >= nbox;
  const BoxDev B = boxes[bad ? 0 : b];
  const int i = pos[3 * s], j = pos[3 * s + 1], k = pos[3 * s + 2];
  bad |= i < 0 || i >= B.n || j < 0 || j >= B.n || k < 0 || k >= B.n;
  const double R = radius[s], nd = ndot[s];
  bad |= !(R > 0.0) || !isfinite(R) || !(nd >= 0.0) || !isfinite(nd) || signbit(nd);
  // traced cells satisfy |Delta|^2 <= floor(R^2); every window cell has
  // |Delta|^2 <= 3 (n/2)^2, so larger limits trace the same set.
  const double cap = 3.0 * (double)(B.n / 2) * (double)(B.n / 2) + 1.0;
  const double rr = fmin(floor(R * R), cap);
  const int r2 = bad ? 0 : (int)rr;
  if (bad) *err = ERR_INPUT;
  const int64_t cell = bad ? 0 : B.off + ((int64_t)i * B.n + j) * B.n + k;
  keys[s] = ((uint64_t)cell << 22) | (uint64_t)r2;
  idx[s] = s;
  r2out[s] = r2;
}

// Number of merged sources and the largest r2, to pinned host memory.
__global__ void k_src_scalars(const int* __restrict__ last_head, const int* __restrict__ last_mid,
                              const int* __restrict__ max_r2, int* __restrict__ out) {
  out[0] = *last_head + *last_mid;
  out[1] = *max_r2;
}

__global__ void k_src_heads(const uint64_t* __restrict__ keys, int nsrc, int* __restrict__ head) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nsrc) return;
  head[t] = (t == 0 || keys[t] != keys[t - 1]) ? 1 : 0;
}

// Merged source m = segment starting at sorted position t: rates summed in
// input order; LPT sort key = (max_r2 - r2) ascending.
__global__ void k_src_merge(const uint64_t* __restrict__ keys, const int* __restrict__ idx,
                            const int* __restrict__ head, const int* __restrict__ mid, int nsrc,
                            const int32_t* __restrict__ pos, const int32_t* __restrict__ box,
                            const double* __restrict__ ndot, const int* __restrict__ r2in,
                            SrcDev* __restrict__ msrc, double* __restrict__ mndot,
                            int* __restrict__ mr2, uint32_t* __restrict__ lkey,
                            int* __restrict__ lval, int* __restrict__ src_of_input, int max_r2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nsrc) return;
  // mid = exclusive scan of head flags: a segment head's own index; any other
  // member sees its head counted already.
  const int m = mid[t] + head[t] - 1;
  src_of_input[idx[t]] = m;  // merged index, remapped to LPT order later
  if (!head[t]) return;
  const int s0 = idx[t];
  double sum = 0.0;
  for (int u = t; u < nsrc && (u == t || !head[u]); ++u) sum += ndot[idx[u]];
  SrcDev d;
  d.i = pos[3 * s0];
  d.j = pos[3 * s0 + 1];
  d.k = pos[3 * s0 + 2];
  d.box = box ? box[s0] : 0;
  msrc[m] = d;
  mndot[m] = sum;
  mr2[m] = r2in[s0];
  lkey[m] = (uint32_t)(max_r2 - r2in[s0]);
  lval[m] = m;
}

// Permute merged sources into LPT order and emit 24 (face, quadrant) items per source.
__global__ void k_src_order(const int* __restrict__ order, int nm, const SrcDev* __restrict__ msrc,
                            const double* __restrict__ mndot, const int* __restrict__ mr2,
                            SrcDev* __restrict__ src, double* __restrict__ ndot,
                            int* __restrict__ r2lim, int* __restrict__ items,
                            int* __restrict__ lpt_of_merged) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nm) return;
  const int m = order[p];
  src[p] = msrc[m];
  ndot[p] = mndot[m];
  r2lim[p] = mr2[m];
  lpt_of_merged[m] = p;
  for (int q = 0; q < 24; ++q) items[24 * p + q] = (p << 5) | q;  // face = q >> 2, quadrant = q & 3
}

__global__ void k_remap(int* __restrict__ a, const int* __restrict__ map, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) a[t] = map[a[t]];
}

static int64_t ball_count(int r2, int n) {
  const int wlo = -(n / 2), whi = (n % 2 == 0) ? n / 2 - 1 : n / 2;
  int64_t cnt = 0;
  const int L = std::min((int)std::floor(std::sqrt((double)r2)) + 1, n);
  for (int a = std::max(-L, wlo); a <= std::min(L, whi); ++a)
    for (int b = std::max(-L, wlo); b <= std::min(L, whi); ++b) {
      const int64_t rem = (int64_t)r2 - (int64_t)a * a - (int64_t)b * b;
      if (rem < 0) continue;
      int w = (int)std::floor(std::sqrt((double)rem));
      while ((int64_t)w * w > rem) --w;
      while ((int64_t)(w + 1) * (w + 1) <= rem) ++w;
      cnt += std::min(w, whi) - std::max(-w, wlo) + 1;
    }
  return cnt;
}

#define CK(x)                                   \
  do {                                          \
    cudaError_t e_ = (x);                       \
    if (e_ != cudaSuccess) {                    \
      st = cuda_fail(e_, #x);                   \
      goto done;                                \
    }                                           \
  } while (0)

void free_sources(Grid& g) {
  Grid::Ingest& w = g.ing;
  dev_free(w.arena);
  cudaFreeHost(w.pinned);
  g.src = nullptr; g.ndot = nullptr; g.r2lim = nullptr; g.items = nullptr;
  g.src_of_input = nullptr; g.ndot_in = nullptr;
  g.src_cap = 0;
  w = Grid::Ingest{};
}

// Grow the per-source arrays (ingest scratch and the ingested sources) to n sources: one
// allocation on the device, and at most one of pinned memory.
static cudaError_t reserve_sources(Grid& g, size_t n) {
  Grid::Ingest& w = g.ing;
  if (n <= w.cap && n <= g.src_cap) return cudaSuccess;
  cudaStreamSynchronize(g.stream);  // earlier work may still read the old arrays
  free_sources(g);
  // CUB scratch for the largest of its uses at n items
  size_t need = 0, tb = 0;
  cudaError_t e = cub::DeviceRadixSort::SortPairs(nullptr, need, w.keys, w.keys2, w.idx, w.idx2,
                                                  (int)n, 0, 64, g.stream);
  tb = std::max(tb, need);
  if (e == cudaSuccess) e = cub::DeviceScan::ExclusiveSum(nullptr, need, w.head, w.mid, (int)n,
                                                          g.stream);
  tb = std::max(tb, need);
  if (e == cudaSuccess) e = cub::DeviceRadixSort::SortPairs(nullptr, need, w.lkey, w.lkey2, w.lval,
                                                            w.order, (int)n, 0, 32, g.stream);
  tb = std::max(tb, need);
  if (e == cudaSuccess) e = cub::DeviceReduce::Max(nullptr, need, w.r2in, w.dscal, (int)n,
                                                   g.stream);
  tb = std::max(tb, need);
  size_t bytes = 0;
  char* base = nullptr;
  auto part = [&](auto*& p, size_t count) {  // (a first pass adds up, a second one places)
    if (base) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(base + bytes);
    bytes += (count * sizeof(*p) + 255) & ~(size_t)255;
  };
  auto parts = [&]() {
    bytes = 0;
    part(w.keys, n); part(w.keys2, n); part(w.idx, n); part(w.idx2, n); part(w.r2in, n);
    part(w.head, n); part(w.mid, n); part(w.msrc, n); part(w.mndot, n); part(w.mr2, n);
    part(w.lkey, n); part(w.lkey2, n); part(w.lval, n); part(w.order, n); part(w.lpt, n);
    part(w.dscal, 4); part(g.src, n); part(g.ndot, n); part(g.r2lim, n); part(g.items, 24 * n);
    part(g.src_of_input, n); part(g.ndot_in, n); part(w.tmp, tb);
  };
  auto pinned = [&]() {
    bytes = 0;
    part(w.r2pin, n);
    if (g.nbox > 1) part(w.srcpin, n);
  };
  if (e == cudaSuccess) {
    parts();
    e = grid_malloc(g, &w.arena, bytes);
    base = w.arena;
    if (base) parts();
  }
  if (e == cudaSuccess) {
    base = nullptr;
    pinned();
    if (bytes <= kPinBytes - 64) {  // behind the grid's own words
      base = reinterpret_cast<char*>(g.pin) + 64;
    } else {
      e = cudaMallocHost(&w.pinned, bytes);
      base = static_cast<char*>(w.pinned);
    }
    if (e == cudaSuccess) pinned();
  }
  if (e != cudaSuccess) {
    free_sources(g);
    return e;
  }
  w.tmp_bytes = tb;
  w.cap = n;
  g.src_cap = n;
  return cudaSuccess;
}

rt_status ingest_sources(Grid& g, int nsrc, const int32_t* d_pos, const int32_t* d_box,
                         const double* d_ndot, const double* d_radius) {
  rt_status st = RT_OK;
  cudaStream_t s = g.stream;
  Grid::Ingest& w = g.ing;
  size_t need = 0;
  int nm = 0;
  const int T = 256;
  const int nb = (nsrc + T - 1) / T;

  g.nsrc = 0; g.nsrc_in = 0; g.max_r2 = 0; g.source_voxels = 0; g.r2_sorted_h.clear();
  if (nsrc == 0) return RT_OK;
  CK(reserve_sources(g, (size_t)nsrc));

  g.pin[0] = 0;
  k_src_keys<<<nb, T, 0, s>>>(g.boxes_d, g.nbox, nsrc, d_pos, d_box, d_ndot, d_radius, w.keys,
                              w.idx, w.r2in, g.pin);
  count_launch();
  CK(cudaGetLastError());
  // stable sort by (cell, r2): co-located sources with equal radius become adjacent
  // (keys of invalid sources are harmless: they are reported below before any use)
  need = w.tmp_bytes;
  CK(cub::DeviceRadixSort::SortPairs(w.tmp, need, w.keys, w.keys2, w.idx, w.idx2, nsrc, 0, 64, s));
  k_src_heads<<<nb, T, 0, s>>>(w.keys2, nsrc, w.head);
  count_launch();
  CK(cudaGetLastError());
  need = w.tmp_bytes;
  CK(cub::DeviceScan::ExclusiveSum(w.tmp, need, w.head, w.mid, nsrc, s));
  need = w.tmp_bytes;
  CK(cub::DeviceReduce::Max(w.tmp, need, w.r2in, w.dscal, nsrc, s));  // for the LPT key
  k_src_scalars<<<1, 1, 0, s>>>(w.head + nsrc - 1, w.mid + nsrc - 1, w.dscal, g.pin + 4);
  count_launch();
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(s));
  if (g.pin[0]) {
    st = fail(RT_ERR_INVALID, "rt_set_sources: source outside its box, bad box id, radius <= 0 "
                              "or non-finite/negative photon rate");
    goto done;
  }
  nm = g.pin[4];
  g.max_r2 = g.pin[5];
  CK(cudaMemcpyAsync(g.ndot_in, d_ndot, nsrc * sizeof(double), cudaMemcpyDeviceToDevice, s));
  k_src_merge<<<nb, T, 0, s>>>(w.keys2, w.idx2, w.head, w.mid, nsrc, d_pos, d_box, d_ndot, w.r2in,
                               w.msrc, w.mndot, w.mr2, w.lkey, w.lval, g.src_of_input, g.max_r2);
  count_launch();
  CK(cudaGetLastError());
  need = w.tmp_bytes;
  CK(cub::DeviceRadixSort::SortPairs(w.tmp, need, w.lkey, w.lkey2, w.lval, w.order, nm, 0, 32, s));
  k_src_order<<<(nm + T - 1) / T, T, 0, s>>>(w.order, nm, w.msrc, w.mndot, w.mr2, g.src, g.ndot,
                                             g.r2lim, g.items, w.lpt);
  count_launch();
  CK(cudaGetLastError());
  k_remap<<<nb, T, 0, s>>>(g.src_of_input, w.lpt, nsrc);
  count_launch();
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(w.r2pin, g.r2lim, nm * sizeof(int), cudaMemcpyDeviceToHost, s));
  if (g.nbox > 1)
    CK(cudaMemcpyAsync(w.srcpin, g.src, nm * sizeof(SrcDev), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  {
    g.r2_sorted_h.assign(w.r2pin, w.r2pin + nm);
    std::map<std::pair<int, int>, int64_t>& memo = g.ball_memo;  // kept between calls
    int64_t sv = 0, last_cnt = 0;
    std::pair<int, int> last_key(-1, -1);
    for (int p = 0; p < nm; ++p) {  // sources come sorted by r2: runs of equal keys
      const int box = g.nbox > 1 ? w.srcpin[p].box : 0;
      const auto key = std::make_pair(g.r2_sorted_h[p], g.boxes_h[box].n);
      if (key != last_key) {
        auto it = memo.find(key);
        if (it == memo.end()) it = memo.emplace(key, ball_count(key.first, key.second)).first;
        last_key = key;
        last_cnt = it->second;
      }
      sv += last_cnt;
    }
    g.source_voxels = sv;
  }
  g.nsrc = nm;
  g.nsrc_in = nsrc;
done:
  return st;
}

// ------------------------------------------------------------ row tables
// Row tables of the unclipped quadrant layers of every distinct R^2 limit: the
// batched trace stages them into shared memory instead of building them per
// item (all 24 items of a source, and all sources with the same limit, share
// them).  Blob of (r2, m): rowpre[0..H+1] (ints: first flat index of row a1,
// then the layer size) and rowof[0..total) (bytes: row of every flat index),
// with H = min(m, isqrt(r2 - m^2)) and row a1 holding a2 = 0..min(H,
// isqrt(r2 - m^2 - a1^2)).
static int isqrt_host(int64_t x) {
  if (x < 0) return -1;
  int r = (int)std::sqrt((double)x);
  while ((int64_t)r * r > x) --r;
  while ((int64_t)(r + 1) * (r + 1) <= x) ++r;
  return r;
}

__global__ void k_row_tables(const int* __restrict__ ent_r2, const int* __restrict__ ent_m,
                             const int* __restrict__ off, unsigned char* __restrict__ rtab,
                             int nent) {
  const int e = blockIdx.x;
  if (e >= nent) return;
  const int m = ent_m[e];
  const int rem = ent_r2[e] - m * m;
  int H = (int)sqrtf((float)rem);
  while (H * H > rem) --H;
  while ((H + 1) * (H + 1) <= rem) ++H;
  H = min(H, m);
  const int nrows = H + 1;
  int* rowpre = reinterpret_cast<int*>(rtab + off[e]);
  unsigned char* rowof = reinterpret_cast<unsigned char*>(rowpre + nrows + 1);
  __shared__ int pre[256 + 1];
  if (threadIdx.x == 0) {
    int run = 0;
    for (int r = 0; r < nrows; ++r) {
      pre[r] = run;
      const int x = rem - r * r;
      int w = (int)sqrtf((float)x);
      while (w * w > x) --w;
      while ((w + 1) * (w + 1) <= x) ++w;
      run += min(H, w) + 1;
    }
    pre[nrows] = run;
  }
  __syncthreads();
  for (int r = threadIdx.x; r <= nrows; r += blockDim.x) rowpre[r] = pre[r];
  for (int r = 0; r < nrows; ++r)
    for (int c = pre[r] + threadIdx.x; c < pre[r + 1]; c += blockDim.x) rowof[c] = (unsigned char)r;
  // zero the padding up to the next 16-byte boundary
  const int used = 4 * (nrows + 1) + pre[nrows];
  for (int b = used + threadIdx.x; b < off[e + 1] - off[e]; b += blockDim.x)
    rtab[off[e] + b] = 0;
}

// Interior row tables of the same layers, for faces traced whole by one warp:
// layer m of a face holds the transverse offsets |t1|, |t2| <= H with
// t1^2 + t2^2 <= r2 - m^2; its interior positions (1 <= a1, a2 <= m-1) form rows
// a1 = 1..LA, LA = min(H, m-1), row a1 holding a2 = 1..min(H, isqrt(r2 - m^2 -
// a1^2), m-1).  Blob: rowpre[0..LA] (ints: first flat index of row r = a1-1,
// then the number of positions) and rowof[0..total) (bytes: row of every flat
// index).  The axes and the rim of the layer are enumerated arithmetically.
__device__ __forceinline__ int isqrt_dev(int x) {
  int w = (int)sqrtf((float)x);
  while (w * w > x) --w;
  while ((w + 1) * (w + 1) <= x) ++w;
  return w;
}

__global__ void k_interior_tables(const int* __restrict__ ent_r2, const int* __restrict__ ent_m,
                                  const int* __restrict__ off, unsigned char* __restrict__ itab,
                                  int nent) {
  const int e = blockIdx.x;
  if (e >= nent) return;
  const int m = ent_m[e];
  const int rem = ent_r2[e] - m * m;
  const int H = min(isqrt_dev(rem), m);
  const int LA = min(H, m - 1);
  int* rowpre = reinterpret_cast<int*>(itab + off[e]);
  unsigned char* rowof = reinterpret_cast<unsigned char*>(rowpre + LA + 1);
  __shared__ int pre[256 + 1];
  if (threadIdx.x == 0) {
    int run = 0;
    for (int r = 0; r < LA; ++r) {
      pre[r] = run;
      const int a1 = r + 1;
      run += max(0, min(min(H, isqrt_dev(rem - a1 * a1)), m - 1));
    }
    pre[LA] = run;
  }
  __syncthreads();
  for (int r = threadIdx.x; r <= LA; r += blockDim.x) rowpre[r] = pre[r];
  for (int r = 0; r < LA; ++r)
    for (int c = pre[r] + threadIdx.x; c < pre[r + 1]; c += blockDim.x) rowof[c] = (unsigned char)r;
  const int used = 4 * (LA + 1) + pre[LA];
  for (int b = used + threadIdx.x; b < off[e + 1] - off[e]; b += blockDim.x)
    itab[off[e] + b] = 0;
}

// Cells of layer m of a whole face as signed offsets (t1, t2), two bytes each, in the
// order that the in-place update of rates.cu needs, last first: the cells off the axes by
// quadrant position (a1, a2), descending rows a1 = H..1 and descending a2 (row a1 holds
// a2 up to min(H, isqrt(r2 - m^2 - a1^2))), the four sign images of a position together
// (they read axis slots, never the other way round); then the axes from a = H inwards,
// (0, a) (0, -a) (a, 0) (-a, 0); the centre is entry 0.  job: (r2, m, offset, cells).
__global__ void k_face_tables(const int4* __restrict__ job, unsigned char* __restrict__ ftab) {
  const int4 q = job[blockIdx.x];
  const int m = q.y;
  const int rem = q.x - m * m;
  const int H = min(isqrt_dev(rem), m);
  char2* out = reinterpret_cast<char2*>(ftab + q.z);
  __shared__ int at[kFaceHcap + 2];  // positions off the axes in rows below a1
  if (threadIdx.x == 0) {
    int run = 0;
    for (int a1 = 1; a1 <= H; ++a1) {
      at[a1] = run;
      run += min(H, isqrt_dev(rem - a1 * a1));
    }
    out[0] = make_char2(0, 0);
  }
  __syncthreads();
  for (int a = 1 + threadIdx.x; a <= H; a += blockDim.x) {
    char2* o = out + 4 * a;
    o[0] = make_char2(0, (signed char)a);
    o[-1] = make_char2(0, (signed char)-a);
    o[-2] = make_char2((signed char)a, 0);
    o[-3] = make_char2((signed char)-a, 0);
  }
  for (int t = threadIdx.x; t < H * H; t += blockDim.x) {
    const int a1 = 1 + t / H, a2 = 1 + t % H;
    if (a2 > min(H, isqrt_dev(rem - a1 * a1))) continue;
    char2* o = out + 4 * H + 1 + 4 * (at[a1] + a2 - 1);
    for (int k = 0; k < 4; ++k)
      o[k] = make_char2((signed char)(k & 1 ? -a1 : a1), (signed char)(k & 2 ? -a2 : a2));
  }
  const int pad = ((2 * q.w + 15) & ~15) / 2 - q.w;
  if (threadIdx.x < pad) out[q.w + threadIdx.x] = make_char2(0, 0);
}

void free_row_tables(Grid& g) {
  dev_free(g.tables);
  g.tables = nullptr;
  g.rtab = nullptr; g.rtab_off = g.rtab_first = g.rtab_hcap = g.rtab_slot = nullptr;
  g.rtab_lay = nullptr;
  g.ftab = nullptr; g.ftab_lay = nullptr;
  g.ftab_bytes = 0;
  g.itab = nullptr; g.itab_off = nullptr;
  g.itab_bytes = 0;
  g.rtab_max_r2 = -1;
  g.rtab_bytes = 0;
  g.rtab_r2s.clear();
  g.rtab_mcap = 0;
}

rt_status ensure_row_tables(Grid& g) {
  rt_status st = RT_OK;
  // distinct limits, descending (r2_sorted_h is in LPT order: descending)
  std::vector<int> r2s;
  for (int v : g.r2_sorted_h)
    if (r2s.empty() || v != r2s.back()) r2s.push_back(v);
  std::sort(r2s.begin(), r2s.end(), std::greater<int>());
  r2s.erase(std::unique(r2s.begin(), r2s.end()), r2s.end());
  const int mcap = g.nmax / 2 + 1;  // no window has more layers
  if (r2s == g.rtab_r2s && mcap == g.rtab_mcap && (g.rtab || r2s.empty())) return RT_OK;
  free_row_tables(g);
  if (r2s.empty()) {
    g.rtab_mcap = mcap;
    return RT_OK;
  }
  std::vector<int4> lay, flay, jobs;
  std::vector<int> square_at(kFaceHcap + 1, -1);
  std::vector<int> ent_r2, ent_m, off, ioff, first(r2s.size()), hcap(r2s.size());
  int64_t cur = 0, icur = 0, fcur = 0;
  int face_stack = 0;
  for (size_t i = 0; i < r2s.size(); ++i) {
    const int v = r2s[i];
    const int L = std::min(isqrt_host(v), mcap);
    first[i] = (int)ent_m.size();
    int hc = 0;
    for (int m = 1; m <= L; ++m) {
      const int64_t rem = (int64_t)v - (int64_t)m * m;
      const int H = std::min(m, isqrt_host(rem));
      const int LA = std::min(H, m - 1);
      int64_t total = 0, itotal = 0;
      int w = isqrt_host(rem);  // of rem - r^2: falls as r grows
      for (int r = 0; r <= H; ++r) {
        while ((int64_t)w * w > rem - (int64_t)r * r) --w;
        total += std::min(H, w) + 1;
        if (r >= 1 && r <= LA) itotal += std::max(0, std::min(std::min(H, w), m - 1));
      }
      hc = std::max(hc, H);
      ent_r2.push_back(v);
      ent_m.push_back(m);
      off.push_back((int)cur);
      ioff.push_back((int)icur);
      lay.push_back(make_int4((int)cur, (int)((4 * (int64_t)(H + 2) + total + 15) & ~(int64_t)15),
                              (int)total, H));
      cur += (4 * (int64_t)(H + 2) + total + 15) & ~(int64_t)15;
      icur += (4 * (int64_t)(LA + 1) + itotal + 15) & ~(int64_t)15;
      if (cur > (int64_t)1 << 30 || H > 254) {  // keep offsets in int, rows in bytes
        g.rtab_r2s = r2s;
        g.rtab_mcap = mcap;
        return RT_OK;  // no tables: the trace builds its own
      }
    }
    hcap[i] = hc;
    // face tables up to the limit's first layer wider than kFaceHcap; layers that are
    // whole squares share one table
    bool wide = false, bwd_fits = true;
    int stack = 0;
    for (int m = 1; m <= L; ++m) {
      const int4 q = lay[first[i] + m - 1];
      wide = wide || q.w > kFaceHcap;
      if (wide) {
        flay.push_back(make_int4(0, 0, 0, 0));
        continue;
      }
      // four images of every position, less those that coincide on the two axes
      const int n = 4 * q.z - 4 * (q.w + 1) + 1;
      const int bytes = (2 * n + 15) & ~15;
      bwd_fits = bwd_fits && q.w <= kBwdFaceHcap;
      if (bwd_fits) stack += n;
      face_stack = std::max(face_stack, stack);
      const bool square = q.z == (m + 1) * (m + 1);
      if (square && square_at[m] >= 0) {
        flay.push_back(make_int4(square_at[m], bytes, n, q.w));
        continue;
      }
      if (square) square_at[m] = (int)fcur;
      jobs.push_back(make_int4(v, m, (int)fcur, n));
      flay.push_back(make_int4((int)fcur, bytes, n, q.w));
      fcur += bytes;
    }
  }
  off.push_back((int)cur);
  ioff.push_back((int)icur);
  const int nent = (int)ent_m.size();
  const int maxv = r2s.front();
  std::vector<int> slot(maxv + 1, -1);
  for (size_t i = 0; i < r2s.size(); ++i) slot[r2s[i]] = (int)i;
  // one allocation: what the host knows (one upload), then the tables the kernels fill
  int *d_r2 = nullptr, *d_m = nullptr;
  int4* d_jobs = nullptr;
  std::vector<char> up;
  size_t bytes = 0;
  auto part = [&](auto*& p, size_t n) {  // (a first pass adds up, a second one places)
    if (g.tables) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(g.tables + bytes);
    bytes += (n * sizeof(*p) + 15) & ~(size_t)15;
  };
  auto host = [&](auto*& p, const auto& v) {
    if (!g.tables) {
      up.resize(bytes + ((v.size() * sizeof(v[0]) + 15) & ~(size_t)15));
      memcpy(up.data() + bytes, v.data(), v.size() * sizeof(v[0]));
    }
    part(p, v.size());
  };
  auto parts = [&]() {
    bytes = 0;
    host(g.rtab_lay, lay); host(g.ftab_lay, flay); host(d_jobs, jobs);
    host(g.rtab_off, off); host(g.itab_off, ioff); host(g.rtab_first, first);
    host(g.rtab_hcap, hcap); host(g.rtab_slot, slot); host(d_r2, ent_r2); host(d_m, ent_m);
    part(g.rtab, cur); part(g.itab, icur); part(g.ftab, fcur + 16);
  };
  cudaStream_t s = g.stream;
#undef CK
#define CK(x)                                   \
  do {                                          \
    cudaError_t e_ = (x);                       \
    if (e_ != cudaSuccess) {                    \
      st = cuda_fail(e_, #x);                   \
      goto fail;                                \
    }                                           \
  } while (0)
  parts();
  CK(grid_malloc(g, &g.tables, bytes));
  parts();
  CK(cudaMemcpyAsync(g.tables, up.data(), up.size(), cudaMemcpyHostToDevice, s));
  if (nent > 0) {
    k_row_tables<<<nent, 64, 0, s>>>(d_r2, d_m, g.rtab_off, g.rtab, nent);
    count_launch();
    CK(cudaGetLastError());
    k_interior_tables<<<nent, 64, 0, s>>>(d_r2, d_m, g.itab_off, g.itab, nent);
    count_launch();
    CK(cudaGetLastError());
    k_face_tables<<<(int)jobs.size(), 64, 0, s>>>(d_jobs, g.ftab);
    count_launch();
    CK(cudaGetLastError());
  }
  CK(cudaStreamSynchronize(s));  // host vectors go out of scope
  g.rtab_max_r2 = maxv;
  g.rtab_bytes = cur;
  g.itab_bytes = icur;
  g.ftab_bytes = fcur;
  g.face_stack = face_stack;
  g.rtab_r2s = r2s;
  g.rtab_mcap = mcap;
  return RT_OK;
fail:
  cudaStreamSynchronize(s);
  free_row_tables(g);
  return st;
#undef CK
}

}  // namespace asora
