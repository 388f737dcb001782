// C ABI of libasora: handles, validation, memory, launches (see include/asora.h).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <cstdlib>
#include <fstream>
#include <mutex>
#include <sstream>
#include <string>
#include <unordered_map>

#include "asora_internal.cuh"
#include "box_limits.h"

namespace asora {

static thread_local std::string g_last_error;
static std::atomic<long long> g_launches{0};

void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

// ---------------------------------------------------------- device memory
static std::mutex g_mem_mutex;
static std::unordered_map<void*, size_t> g_mem_sizes;
static int64_t g_mem_live = 0;
static int64_t g_mem_limit = -1;  // -1: not read yet, 0: no limit

static int64_t mem_limit_locked() {
  if (g_mem_limit < 0) {
    g_mem_limit = 0;
    if (const char* v = std::getenv("ASORA_DEVICE_MEMORY_LIMIT")) {
      char* end = nullptr;
      const long long x = std::strtoll(v, &end, 10);
      if (end != v && x > 0) g_mem_limit = x;
    }
  }
  return g_mem_limit;
}

cudaError_t dev_malloc_raw(void** p, size_t bytes) {
  *p = nullptr;
  std::lock_guard<std::mutex> lk(g_mem_mutex);
  const int64_t lim = mem_limit_locked();
  if (lim > 0 && g_mem_live + (int64_t)bytes > lim) return cudaErrorMemoryAllocation;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    *p = nullptr;
    return e;
  }
  g_mem_sizes[*p] = bytes;
  g_mem_live += (int64_t)bytes;
  return cudaSuccess;
}

cudaError_t dev_free(void* p) {
  if (!p) return cudaSuccess;
  {
    std::lock_guard<std::mutex> lk(g_mem_mutex);
    auto it = g_mem_sizes.find(p);
    if (it != g_mem_sizes.end()) {
      g_mem_live -= (int64_t)it->second;
      g_mem_sizes.erase(it);
    }
  }
  return cudaFree(p);
}

rt_status fail(rt_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

rt_status cuda_fail(cudaError_t e, const char* what) {
  g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
  cudaGetLastError();  // clear a sticky-free error so the next call starts clean
  return e == cudaErrorMemoryAllocation ? RT_ERR_OOM : RT_ERR_CUDA;
}

// Whether work given to the stream now is captured into a caller's graph (if in doubt: yes).
static bool in_capture(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  const bool clear = cudaPeekAtLastError() == cudaSuccess;
  if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st != cudaStreamCaptureStatusNone;
  if (clear) cudaGetLastError();  // (an error that was there stays)
  return true;
}

bool release_scratch(Grid& g) {
  if (!g.od_scratch || g.od_captured || in_capture(g.stream)) return false;
  cudaGetLastError();  // (of the allocation that failed)
  dev_free(g.od_scratch);  // waits for what still uses it
  g.od_scratch = nullptr;
  ++g.epoch;  // a kept graph holds its address
  return true;
}

static int isqrt_h(int64_t x) {
  if (x <= 0) return 0;
  int64_t r = (int64_t)std::sqrt((double)x);
  while (r * r > x) --r;
  while ((r + 1) * (r + 1) <= x) ++r;
  return (int)r;
}

static void free_grid(Grid* g) {
  dev_free(g->small); cudaFreeHost(g->pin); dev_free(g->gtab); dev_free(g->htab);
  dev_free(g->dtau); dev_free(g->dtauT); dev_free(g->invn);
  free_sources(*g);
  dev_free(g->geo); dev_free(g->georow); dev_free(g->kap);
  dev_free(g->cube); dev_free(g->od_scratch); dev_free(g->xbuf); dev_free(g->xavg);
  dev_free(g->xavg2); dev_free(g->xhi_int);
  dev_free(g->bwd_stack); dev_free(g->dq_merged); dev_free(g->bwd_redo);
  free_row_tables(*g);
  if (g->it_exec) cudaGraphExecDestroy(g->it_exec);
  if (g->it_stream) cudaStreamDestroy(g->it_stream);
  for (auto& e : g->ev)
    if (e) cudaEventDestroy(e);
  delete g;
}

#define TRY(x)                                      \
  do {                                              \
    cudaError_t e_ = (x);                           \
    if (e_ != cudaSuccess) return cuda_fail(e_, #x); \
  } while (0)

// Cell-size dependent constants of a box record.
static void set_box_cell(BoxDev& B, double c, double sigma0) {
  B.cell = c;
  B.inv_cell3 = 1.0 / (c * c * c);
  B.thin_fac = sigma0 / (c * c);
  B.sig_cell = sigma0 * c;
}

static rt_status ensure_geometry(Grid& g, int mmax) {
  if (mmax <= g.geo_mmax) return RT_OK;
  GeoEntry* geo = nullptr;
  GeoRow* georow = nullptr;
  TRY(grid_malloc(g, &geo, geo_count(mmax) * sizeof(GeoEntry)));
  const int kmax = std::min(mmax, kKapMax);
  double* kap = nullptr;
  const size_t nkap = 4 * georow_count(kmax) + (size_t)(kmax + 1) * (kmax + 2);
  cudaError_t e = grid_malloc(g, &georow, georow_count(mmax) * sizeof(GeoRow));
  if (e == cudaSuccess) e = grid_malloc(g, &kap, nkap * sizeof(double));
  if (e == cudaSuccess) e = launch_geometry(geo, georow, kap, g.p.tau_lim, mmax, g.stream);
  if (e != cudaSuccess) {
    dev_free(geo);
    dev_free(georow);
    dev_free(kap);
    return cuda_fail(e, "geometry");
  }
  dev_free(g.geo);
  dev_free(g.georow);
  dev_free(g.kap);
  g.geo = geo;
  g.georow = georow;
  g.kap = kap;
  g.geo_mmax = mmax;
  g.kap_mmax = kmax;
  return RT_OK;
}

// Largest layer half-width min(m, floor(sqrt(r2 - m^2))) over the layers of a face (at
// least 1): m grows up to sqrt(r2 / 2), beyond which the square root is the smaller.
static int face_hcap(int r2, int nmax) {
  return std::max(1, std::min({isqrt_h(r2), nmax / 2 + 1, isqrt_h(r2 / 2)}));
}

static TraceArgs base_args(Grid& g) {
  TraceArgs a{};
  a.boxes = g.boxes_d;
  a.dtau = g.dtau;
  a.dtauT = g.dtauT;
  a.invn = g.invn;
  a.thick = g.invn;
  a.src = g.src;
  a.ndot = g.ndot;
  a.r2lim = g.r2lim;
  a.queue = g.queue;
  a.geo = g.geo;
  a.georow = g.georow;
  a.rtab = g.rtab;
  a.rtab_off = g.rtab_off;
  a.rtab_first = g.rtab_first;
  a.rtab_hcap = g.rtab_hcap;
  a.rtab_slot = g.rtab_slot;
  a.rtab_max_r2 = g.rtab_max_r2;
  a.rtab_lay = g.rtab_lay;
  a.ftab = g.ftab;
  a.ftab_lay = g.ftab_lay;
  a.itab = g.itab;
  a.itab_off = g.itab_off;
  a.neg_zero = -0.0;
  a.interp_mode = g.interp_mode;
  a.tau_w0 = g.tau_w0;
  a.geo_mmax = g.geo_mmax;
  a.kap = g.kap;
  a.kap_mmax = g.kap_mmax;
  a.kappa = g.kap ? g.kap + georow_count(g.kap_mmax) : nullptr;
  a.ikappa = g.kap ? g.kap + 2 * georow_count(g.kap_mmax) : nullptr;
  a.dsik = g.kap ? g.kap + 3 * georow_count(g.kap_mmax) : nullptr;
  a.tab.g = g.gtab;
  a.tab.h = g.htab;
  a.tab.kind = g.tab_kind;
  a.tab.E0 = g.E0;
  a.tab.B = g.B;
  if (g.tab_kind == RT_TABLE_GREY_EXACT) {
    // exp(-tau) is exactly 0 in double beyond tau = 746; skip the rate there
    const double lim = 750.0;
    std::memcpy(&a.tab.tau_max_bits, &lim, 8);
    a.tab.tau_min_bits = 0;
  } else {
    const double tmin = std::ldexp(1.0, -g.E0), tmax = std::ldexp(1.0, g.E1);
    std::memcpy(&a.tab.tau_min_bits, &tmin, 8);
    std::memcpy(&a.tab.tau_max_bits, &tmax, 8);
  }
  a.tau_lim = g.p.tau_lim;
  a.sigma0 = g.p.sigma0_cm2;
  a.err = g.err;
  a.rate_cells = g.counters;
  {
    double tmax;
    std::memcpy(&tmax, &a.tab.tau_max_bits, 8);
    const double bound = tmax * (1.0 + std::ldexp(1.0, -40));
    std::memcpy(&a.exit_bits, &bound, 8);
  }
  a.early_exit = 0;
  return a;
}

// Synchronises the grid's stream; error bits latched by the kernels since the last check,
// cleared.
static rt_status latched_errors(Grid& g) {
  TRY(cudaMemcpyAsync(g.pin + 1, g.err, sizeof(int), cudaMemcpyDeviceToHost, g.stream));
  TRY(cudaStreamSynchronize(g.stream));
  const int herr = g.pin[1];
  if (!herr) return RT_OK;
  TRY(cudaMemsetAsync(g.err, 0, sizeof(int), g.stream));
  TRY(cudaStreamSynchronize(g.stream));
  std::string what;
  if (herr & ERR_LAYER_CAP) what += " layer wider than the shared-memory capacity;";
  if (herr & ERR_GEO) what += " layer beyond the geometry table;";
  if (herr & ERR_CUBE) what += " source extent beyond the plain schedule's cube;";
  if (herr & ERR_INPUT) what += " invalid input data;";
  return fail(RT_ERR_BOUNDS, "device-side check failed (error bits " + std::to_string(herr) +
                                 "):" + what + " the results of the last trace are incomplete");
}

static rt_status check_ready(Grid& g, const char* who) {
  if (!g.have_tables) return fail(RT_ERR_STATE, std::string(who) + ": rt_set_tables not called");
  if (!g.nH) return fail(RT_ERR_STATE, std::string(who) + ": rt_set_density not called");
  if (!g.xHI) return fail(RT_ERR_STATE, std::string(who) + ": rt_set_xHI not called");
  return RT_OK;
}

// Scratch cubes of the plain schedule for nsrc sources.
constexpr int kPlainBlock = 256;
static rt_status ensure_cube(Grid& g, int nsrc, int* out_grid, int* out_E) {
  const int E = std::max(1, std::min(isqrt_h(g.max_r2), g.nmax / 2));
  const int grid = std::min(nsrc, std::max(1, shells_max_grid(kPlainBlock)));
  const size_t side = 2 * (size_t)E + 1;
  const size_t need = side * side * side * sizeof(double) * (size_t)grid;
  if (need > g.cube_bytes) {
    dev_free(g.cube);
    g.cube = nullptr;
    g.cube_bytes = 0;
    TRY(grid_malloc(g, &g.cube, need));
    g.cube_bytes = need;
  }
  *out_grid = grid;
  *out_E = E;
  return RT_OK;
}

// First source (LPT order) whose layers fit half-width hlim; ns: none.
static int first_fitting(const Grid& g, const int* r2s, int ns, int hlim) {
  if (hlim <= 0) return ns;
  int lo = 0, hi = ns;
  while (lo < hi) {
    const int mid = (lo + hi) / 2;
    if (face_hcap(r2s[mid], g.nmax) <= hlim) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Threads of a CTA that has an SM to itself, for layers of half-width h.  One source, us
// a pass with 128 / 256 / 512 threads (column densities; rates in an ionised box): R = 16
// (h = 11) 50 / 50 / 52; 51 / 54 / 55; R = 24 (16) 70 / 66 / 68; 83 / 76 / 79; R = 40 (28)
// 168 / 137 / 133; 223 / 176 / 169; R = 70 (49) 566 / 382 / 321; 881 / 537 / 454.
static int few_items_block(int h) { return (h < 12 ? 128 : h < 24 ? 256 : 512) | kAhead; }

// How much longer a warp would take for one of `parts` equal parts of the widest source's
// ball than all work takes the GPU's resident warps (16 per SM at the larger widths).
static double longest_part(const Grid& g, int parts) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const double r = std::sqrt((double)g.max_r2);
  const double ball = std::min(4.18879 * r * r * r, (double)g.nmax * g.nmax * g.nmax);
  return ball / parts * (16.0 * sms) / std::max(1.0, (double)g.source_voxels);
}

// Launches of the batched rates: sources [cut[k], cut[k+1]) (LPT order) by CTAs of
// mode[0] threads (k = 0) or by warps with one quadrant, two, or a whole face (k > 0).
struct RatesPlan {
  static constexpr int kClasses = 6;
  int mode[kClasses] = {128, 1, 1, 2, 4, 4};
  int cut[kClasses + 1] = {};
};

// With rt_set_schedule (or an autotuned choice): its thresholds.  Otherwise by rule.
// Measured on uniform catalogues (batched trace, ms: CTA of 128 / one quadrant per warp
// / two / a face; 128^3): R = 12 (half-width 8), 4e4 sources 16.7 / 10.4 / 7.3 / 5.2;
// R = 22 (15), 1e4: 7.4 / 4.7 / 4.0 / 3.7; R = 27 (19), 8e3: 7.7 / 5.1 / 4.7 / 5.8;
// R = 33 (23), 5e3: 6.5 / 4.8 / 4.6 / -; R = 50 (35), 2e3: 5.8 / 5.3 / 7.0 / -; R = 60
// (42), 1e3: 4.8 / 5.3 / - / -: hence the half-widths, but for two quadrants: since one
// runs up to 24 warps per SM it takes at R = 33 what two take (4.22 / 4.28), in an ionised box
// (1.5e3 sources) 4.88 / 5.62, with the early exit 0.41 / 0.45; at R = 27 5.17 / 5.03, 5.51 /
// 5.57 and 0.75 / 0.71.  With optical-depth weights two never pay (2e3 sources of R =
// 5..50: 2.77 ms with them, 2.54 without).  One quadrant per warp is launched twice, as
// its warps' shared memory goes by the widest source: from
// half-width 30 on 14 warps fit an SM, below 21 (250^3, 3e5 sources of R = 5..50: 143.4 /
// 138.2 ms in four launches; 128^3, 1.6e4 7.26 / 7.21; 64^3, 1e3 0.47 / 0.54: only where
// both parts are large); so are faces, from half-width 14 on (15 warps, below 21: 139.1 /
// 135.9 ms; the 64-box ensemble 18.7 / 18.1; 250^3, 1e5 with the early exit 5.18 / 5.03).  A launch pays for its last
// wave, so where several classes would be launched a class of few items joins the finer
// one before it (64^3, 1e3 sources of R = 5..50: one launch 0.52, three 0.87 ms), and two
// quadrants per warp take many (128^3, two / one, batched and with the early exit: 900
// sources of R = 27 0.542 / 0.520 and 0.204 / 0.141; 3e3 1.57 / 1.59 and 0.284 / 0.237), and
// where one quadrant would take a warp longer than all work takes the GPU, CTAs trace
// everything (64^3, 10 sources of R = 20: 0.048 against 0.057 ms; 128^3, 40 of R = 40:
// 0.123 / 0.187).  With at most two items per SM they are the kAhead ones; with up to
// four, CTAs of 256 pay for wide layers (200^3, 20 sources of R = 45: 0.146 / 0.177;
// 128^3, 40 of R = 40, six items per SM: 0.156 / 0.128).  With the early exit an item
// ends after a few layers and a wide one's latency counts: in a catalogue whose widest
// quadrant takes a tenth of the whole, CTAs from half-width 20 on (128^3, early exit, CTA /
// one quadrant, ms: 500 sources of R = 30 0.42 / 0.57 or 0.095 / 0.150 by cell size; 100
// of R = 40 0.115 / 0.236; but 500 of R = 12 0.099 / 0.083).
static RatesPlan rates_plan(const Grid& g, const int* r2s, int ns, bool exit) {
  RatesPlan p;
  p.mode[0] = g.block_big;
  constexpr int K = RatesPlan::kClasses;
  p.cut[K] = ns;
  if (g.explicit_schedule) {
    p.cut[1] = first_fitting(g, r2s, ns, g.hsmall);
    for (int k = 2; k < K; ++k)
      p.cut[k] = g.ftab ? std::max(p.cut[1], first_fitting(g, r2s, ns, g.hface)) : ns;
    return p;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const double warps = 16.0 * sms;  // resident at the larger half-widths
  p.mode[0] = 128;
  if (longest_part(g, 24) > 1.2) {
    const int h = face_hcap(r2s[0], g.nmax);
    if (24 * ns <= 2 * sms) p.mode[0] = few_items_block(h);
    else if (24 * ns <= 4 * sms && h >= 24) p.mode[0] = 256;
    for (int k = 1; k < K; ++k) p.cut[k] = ns;
    return p;
  }
  const int face = g.ftab ? 16 : 0, small = g.ftab ? 13 : 0;
  const bool od = g.interp_mode == RT_INTERP_OPTICAL_DEPTH;
  if (od) p.mode[3] = 1;
  const int lim[K] = {0, exit && longest_part(g, 24) > 0.1 ? 19 : 38, 30, od ? face : 20, face,
                      small};
  for (int k = 1; k < K; ++k) p.cut[k] = std::max(p.cut[k - 1], first_fitting(g, r2s, ns, lim[k]));
  for (int k = K - 1; k > 1; --k) {
    double items = 24.0 / p.mode[k] * (p.cut[k + 1] - p.cut[k]);
    if (p.mode[k] == p.mode[k - 1])
      items = std::min(items, 24.0 / p.mode[k] * (p.cut[k] - p.cut[k - 1])) / 2;
    const double least = p.mode[k] == 2 ? (exit ? 30 : 8) : p.cut[k] > 0 ? 6 : 1.2;
    if (items < least * warps) p.cut[k] = p.cut[k + 1];
  }
  return p;
}

// Whether the batched rates go to rates.cu (its precompute: zeros for the thick terms).
// With optical-depth-modulated weights only its warps do; what needs CTAs takes trace.cu.
static bool takes_rates_kernels(const Grid& g, bool exit) {
  if (g.interp_mode == RT_INTERP_GEOMETRIC) return true;
  return g.nsrc > 0 && g.od_scratch && rates_plan(g, g.r2_sorted_h.data(), g.nsrc, exit).cut[1] == 0;
}

struct RatesLaunch {
  int mode, hcap, begin, end, grid, wpb;  // items [begin, end)
  size_t smem;
};
static rt_status rates_launches(Grid& g, bool exit, std::vector<RatesLaunch>& out) {
  const int* r2s = g.r2_sorted_h.data();
  const RatesPlan plan = rates_plan(g, r2s, g.nsrc, exit);
  const bool od = g.interp_mode == RT_INTERP_OPTICAL_DEPTH;
  for (int k = 0; k < RatesPlan::kClasses; ++k) {
    if (plan.cut[k + 1] <= plan.cut[k]) continue;
    RatesLaunch L;
    L.mode = plan.mode[k];
    L.hcap = face_hcap(r2s[plan.cut[k]], g.nmax);
    const int per = k == 0 ? 24 : 24 / L.mode;
    L.begin = per * plan.cut[k];
    L.end = per * plan.cut[k + 1];
    L.smem = rates_smem_bytes(L.hcap, L.mode);
    if (L.smem > 227 * 1024)
      return fail(RT_ERR_INVALID, "rt_raytrace: radius too large for the batched schedule's "
                                  "shared-memory layers; use RT_SCHED_PLAIN");
    L.wpb = 1;
    // (kept per grid: what fits an SM does not change, and asking takes 10 us a trace)
    const std::array<int, 4> key{L.mode, L.hcap, exit, od};
    auto fits = g.occupancy.find(key);
    if (fits == g.occupancy.end()) {
      int maxg = 0;
      if (k == 0) {
        maxg = rates_max_grid(L.mode, L.smem, 1, exit, od);
      } else {
        // CTAs of as many warps as keeps the most resident (a warp's shared memory grows
        // with its layer capacity, and every CTA also reserves some; ties go to the
        // larger CTA)
        for (int cand = rates_max_warps(L.mode, exit, od); cand >= 1; --cand) {
          const int mg = rates_max_grid(L.mode, L.smem * cand, cand, exit, od);
          if (mg * cand > maxg * L.wpb) {
            maxg = mg;
            L.wpb = cand;
          }
        }
      }
      if (maxg > 0) fits = g.occupancy.emplace(key, std::make_pair(maxg, L.wpb)).first;
    }
    const int maxg = fits == g.occupancy.end() ? 0 : fits->second.first;
    if (maxg > 0) L.wpb = fits->second.second;
    if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace: no occupancy for a rate kernel");
    const int n = L.end - L.begin;
    L.grid = L.mode & kAhead ? n : std::max(1, std::min((n + L.wpb - 1) / L.wpb, maxg));
    L.smem *= L.wpb;
    out.push_back(L);
  }
  return RT_OK;
}

static rt_status run_rates(Grid& g, const TraceArgs& a, const int* items) {
  std::vector<RatesLaunch> ls;
  rt_status st = rates_launches(g, a.early_exit != 0, ls);
  if (st != RT_OK) return st;
  for (size_t k = 0; k < ls.size(); ++k) {
    const RatesLaunch& L = ls[k];
    TraceArgs b = a;
    b.items = items;
    b.hcap = L.hcap;
    b.item_begin = L.begin;
    b.n_items = L.end;
    b.queue = g.queue + k;
    b.scratch = g.od_scratch;
    TRY(launch_rates(g, b, L.mode, L.grid, L.smem, L.wpb));
    if (++g.stats.launches == 1) {
      g.stats.block = L.mode <= 4 ? 32 * L.wpb : L.mode & ~kAhead;
      g.stats.grid = L.grid;
    }
  }
  return RT_OK;
}

// Trace all sources, adding rates into `gamma` (already zeroed) or writing one
// source's column densities.  `items`/`n_items` select the work.
// single_r2 >= 0: the items are the 24 of one source with that R^2 limit (else
// the grid's LPT list, whose limits are g.r2_sorted_h).
static rt_status run_trace(Grid& g, double* gamma, double* coldens, const int* items, int n_items,
                           int schedule, int nsrc_plain, const int* skip = nullptr,
                           bool early_exit = false, int single_r2 = -1) {
  TraceArgs a = base_args(g);
  a.gamma = gamma;
  a.coldens = coldens;
  a.skip = skip;
  a.early_exit = early_exit ? 1 : 0;
  g.stats.launches = 0;
  TRY(cudaMemsetAsync(g.counters, 0, 64 + 8 * sizeof(int), g.stream));  // and the queues
  const bool od = a.interp_mode == RT_INTERP_OPTICAL_DEPTH;
  const bool rates = gamma && takes_rates_kernels(g, early_exit);
  if (schedule != RT_SCHED_PLAIN && g.nmax > kMaxBox32)
    return fail(RT_ERR_INVALID, "rt_raytrace: the batched schedule needs boxes of at most "
                                "1290^3 cells (32-bit offsets); use RT_SCHED_PLAIN");
  if (schedule == RT_SCHED_PLAIN) {
    const int block = kPlainBlock;
    int grid = 0, E = 0;
    rt_status cs = ensure_cube(g, nsrc_plain, &grid, &E);
    if (cs != RT_OK) return cs;
    a.scratch = g.cube;
    a.hcap = E;
    a.items = items;
    a.n_items = nsrc_plain;
    TRY(launch_trace_shells(g, a, block, grid));
    g.stats.block = block;
    g.stats.grid = grid;
    g.stats.launches = 1;
    g.stats.items = nsrc_plain;
  } else if (rates) {
    rt_status rs = run_rates(g, a, items);
    if (rs != RT_OK) return rs;
    TRY(launch_add_thick(g, gamma, skip));
    g.stats.items = n_items;
  } else {
    // Batched: items of large sources are traced by whole CTAs, items whose
    // layers fit g.hsmall by single warps, and the faces of sources whose layers
    // fit g.hface by single warps that trace a face whole.  Items come
    // in LPT order (24 per source, r2 non-increasing), so each mode gets a
    // contiguous range of sources: [0, pw) CTAs, [pw, p4) warps, [p4, ns) whole faces.
    const int* r2s = single_r2 >= 0 ? &single_r2 : g.r2_sorted_h.data();
    const int ns = n_items / 24;
    const int pw = first_fitting(g, r2s, ns, g.hsmall);
    const int p4 = std::max(pw, first_fitting(g, r2s, ns, g.hface));
    const int hbig = face_hcap(r2s[0], g.nmax);
    a.items = items;
    g.stats.launches = 0;
    // warp modes: CTAs of 1..8 warps, whichever keeps the most warps resident (a
    // warp's shared memory grows with its layer capacity, and every CTA also
    // reserves some; ties go to the larger CTA)
    auto warp_launch = [&](int mode, int hcap, int item_begin, int item_end, int* queue) {
      const size_t smem = faces_smem_bytes(hcap, mode, od);
      int wpb = 8, maxg = 0;
      for (int cand = 8; cand >= 1; --cand) {
        const int mg = faces_max_grid(mode, smem * cand, cand, od);
        if (mg * cand > maxg * wpb) {
          maxg = mg;
          wpb = cand;
        }
      }
      if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace: no occupancy for a warp face kernel");
      g.warps_per_block = wpb;
      TraceArgs b = a;
      b.hcap = hcap;
      b.item_begin = item_begin;
      b.n_items = item_end;
      b.queue = queue;
      const int nitem = item_end - item_begin;
      const int grid = std::max(1, std::min((nitem + wpb - 1) / wpb, maxg));
      TRY(launch_trace_faces(g, b, mode, grid, smem * wpb, wpb));
      g.stats.launches += 1;
      if (g.stats.launches == 1) {
        g.stats.block = 32 * wpb;
        g.stats.grid = grid;
      }
      return RT_OK;
    };
    if (pw > 0) {
      const int block = g.block_big;
      const size_t smem = faces_smem_bytes(hbig, block, od);
      if (smem > 227 * 1024)
        return fail(RT_ERR_INVALID, "rt_raytrace: radius too large for the batched schedule's "
                                    "shared-memory layers; use RT_SCHED_PLAIN");
      const int maxg = faces_max_grid(block, smem, 8, od);
      if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace: no occupancy for the face kernel");
      TraceArgs b = a;
      b.hcap = hbig;
      b.item_begin = 0;
      b.n_items = 24 * pw;
      b.queue = g.queue;
      const int grid = std::max(1, std::min(b.n_items, maxg));
      TRY(launch_trace_faces(g, b, block, grid, smem));
      g.stats.block = block;
      g.stats.grid = grid;
      g.stats.launches += 1;
    }
    if (p4 > pw) {
      rt_status ws = warp_launch(32, face_hcap(r2s[pw], g.nmax), 24 * pw, 24 * p4, g.queue + 1);
      if (ws != RT_OK) return ws;
    }
    if (ns > p4) {  // whole faces: face items it -> items[4 it]
      rt_status ws = warp_launch(4, face_hcap(r2s[p4], g.nmax), 6 * p4, 6 * ns, g.queue + 2);
      if (ws != RT_OK) return ws;
    }
    g.stats.items = n_items;
  }
  g.stats.schedule = schedule;
  return RT_OK;
}

}  // namespace asora

using namespace asora;

extern "C" {

void rt_params_default(rt_params* p) {
  if (!p) return;
  p->sigma0_cm2 = 6.30e-18;
  p->tau_lim = 1e-7;
}

const char* rt_last_error(void) { return g_last_error.c_str(); }

long long rt_kernel_launch_count(void) { return g_launches.load(); }

rt_status rt_ensemble_create(rt_grid_t* out, int nbox, const int* h_n, const double* h_cell_cm,
                             const rt_params* p, rt_stream_t s) {
  if (!out) return fail(RT_ERR_INVALID, "rt_ensemble_create: null handle pointer");
  *out = nullptr;
  if (nbox < 1 || nbox > (1 << 20) || !h_n || !h_cell_cm)
    return fail(RT_ERR_INVALID, "rt_ensemble_create: bad box list");
  rt_params prm;
  rt_params_default(&prm);
  if (p) prm = *p;
  if (!(prm.sigma0_cm2 > 0) || !std::isfinite(prm.sigma0_cm2) || !(prm.tau_lim >= 0) ||
      !std::isfinite(prm.tau_lim))
    return fail(RT_ERR_INVALID, "rt_ensemble_create: bad parameters");
  Grid* g = new Grid;
  g->p = prm;
  g->stream = (cudaStream_t)s;
  g->nbox = nbox;
  int64_t off = 0;
  for (int b = 0; b < nbox; ++b) {
    const int n = h_n[b];
    const double c = h_cell_cm[b];
    if (n < 1 || n > 4096 || !(c > 0) || !std::isfinite(c)) {
      delete g;
      return fail(RT_ERR_INVALID, "rt_ensemble_create: box size must be 1..4096 and cell > 0");
    }
    BoxDev B;
    B.n = n;
    B.wlo = -(n / 2);
    B.whi = (n % 2 == 0) ? n / 2 - 1 : n / 2;
    B.off = off;
    set_box_cell(B, c, prm.sigma0_cm2);
    g->boxes_h.push_back(B);
    g->cell_comoving.push_back(c);
    off += (int64_t)n * n * n;
    g->nmax = std::max(g->nmax, n);
  }
  g->ncell = off;
  cudaError_t e = cudaSuccess;
  e = dev_malloc(&g->dtau, g->ncell * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&g->dtauT, g->ncell * sizeof(double));
  if (e == cudaSuccess) e = dev_malloc(&g->invn, g->ncell * sizeof(double));
  // the small arrays: counters 0 (8), queue 64 (64 ints: the counters and the first 8 are
  // cleared together), err 320, flags 384 (16 ints), unconv 448 (16 64-bit counts), boxes 576
  const size_t small = 576 + nbox * sizeof(BoxDev);
  if (e == cudaSuccess) e = dev_malloc(&g->small, small);
  if (e == cudaSuccess) {
    g->counters = reinterpret_cast<unsigned long long*>(g->small);
    g->queue = reinterpret_cast<int*>(g->small + 64);
    g->err = reinterpret_cast<int*>(g->small + 320);
    g->flags = reinterpret_cast<int*>(g->small + 384);
    g->unconv = reinterpret_cast<int64_t*>(g->small + 448);
    g->boxes_d = reinterpret_cast<BoxDev*>(g->small + 576);
    std::vector<char> up(small, 0);
    memcpy(up.data() + 576, g->boxes_h.data(), nbox * sizeof(BoxDev));
    e = cudaMemcpy(g->small, up.data(), small, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&g->pin), kPinBytes);
  for (auto& ev : g->ev)
    if (e == cudaSuccess) e = cudaEventCreate(&ev);
  if (e != cudaSuccess) {
    rt_status st = cuda_fail(e, "rt_ensemble_create");
    free_grid(g);
    return st;
  }
  *out = reinterpret_cast<rt_grid_t>(g);
  return RT_OK;
}

rt_status rt_grid_create(rt_grid_t* out, int n, double cell_cm, const rt_params* p, rt_stream_t s) {
  return rt_ensemble_create(out, 1, &n, &cell_cm, p, s);
}

rt_status rt_set_stream(rt_grid_t h, rt_stream_t s) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_stream: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  g.stream = (cudaStream_t)s;
  ++g.epoch;
  return RT_OK;
}

rt_status rt_set_tables(rt_grid_t h, int kind, int E0, int E1, int bits, const double* h_g,
                        const double* h_h) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_tables: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  const int K = rt_table_nknots(E0, E1, bits);
  if (K < 0 || E0 > 1000 || E1 > 1000 || bits > 10)
    return fail(RT_ERR_INVALID, "rt_set_tables: need 1 <= E0,E1 <= 1000 and 0 <= bits <= 10");
  if (kind != RT_TABLE_CHORDS && kind != RT_TABLE_GREY_EXACT)
    return fail(RT_ERR_INVALID, "rt_set_tables: unknown table kind");
  const int S = K - 1;
  std::vector<double2> gc(S), hc(S);
  if (kind == RT_TABLE_CHORDS) {
    if (!h_g || !h_h) return fail(RT_ERR_INVALID, "rt_set_tables: knot arrays required");
    for (int k = 0; k < K; ++k)
      if (!std::isfinite(h_g[k]) || !std::isfinite(h_h[k]) || h_g[k] < 0 || h_h[k] < 0)
        return fail(RT_ERR_INVALID, "rt_set_tables: knot values must be finite and >= 0");
    auto tau = [&](int idx) {
      if (idx == 0) return 0.0;
      if (idx == K - 1) return std::ldexp(1.0, E1);
      const int t = idx - 1;
      return std::ldexp(1.0 + (double)(t & ((1 << bits) - 1)) / (double)(1 << bits), (t >> bits) - E0);
    };
    for (int s = 0; s < S; ++s) {
      const double tl = tau(s), th = tau(s + 1);
      double c1 = (h_g[s + 1] - h_g[s]) / (th - tl);
      gc[s] = make_double2(std::fma(-c1, tl, h_g[s]), c1);
      c1 = (h_h[s + 1] - h_h[s]) / (th - tl);
      hc[s] = make_double2(std::fma(-c1, tl, h_h[s]), c1);
    }
  }
  double2 *dg = nullptr, *dh = nullptr;
  TRY(grid_malloc(g, &dg, S * sizeof(double2)));
  cudaError_t e = grid_malloc(g, &dh, S * sizeof(double2));
  if (e == cudaSuccess) e = cudaMemcpy(dg, gc.data(), S * sizeof(double2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dh, hc.data(), S * sizeof(double2), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    dev_free(dg);
    dev_free(dh);
    return cuda_fail(e, "rt_set_tables");
  }
  dev_free(g.gtab);
  dev_free(g.htab);
  g.gtab = dg;
  g.htab = dh;
  g.tab_kind = kind;
  g.E0 = E0;
  g.E1 = E1;
  g.B = bits;
  g.have_tables = true;
  ++g.epoch;
  return RT_OK;
}

static rt_status set_field(rt_grid_t h, const double* d, bool density) {
  const char* who = density ? "rt_set_density" : "rt_set_xHI";
  if (!h) return fail(RT_ERR_INVALID, std::string(who) + ": null grid");
  if (!d) return fail(RT_ERR_INVALID, std::string(who) + ": null field");
  Grid& g = *reinterpret_cast<Grid*>(h);
  g.pin[0] = 0;
  TRY(launch_validate_field(g, d, density ? 1e12 : 1.0));
  TRY(cudaStreamSynchronize(g.stream));
  if (g.pin[0])
    return fail(RT_ERR_INVALID, density ? "rt_set_density: n_H must be finite, >= +0 and <= 1e12"
                                        : "rt_set_xHI: x_HI must lie in [+0, 1]");
  if (density) g.nH = d; else g.xHI = d;
  ++g.epoch;
  return RT_OK;
}

rt_status rt_set_scale_factor(rt_grid_t h, double a) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_scale_factor: null grid");
  if (!(a > 0.0) || !std::isfinite(a) || a > 1e6 || a < 1e-6)
    return fail(RT_ERR_INVALID, "rt_set_scale_factor: a must be finite and in [1e-6, 1e6]");
  Grid& g = *reinterpret_cast<Grid*>(h);
  g.a = a;
  g.inv_a3 = 1.0 / (a * a * a);
  for (int b = 0; b < g.nbox; ++b) set_box_cell(g.boxes_h[b], g.cell_comoving[b] * a, g.p.sigma0_cm2);
  TRY(cudaMemcpyAsync(g.boxes_d, g.boxes_h.data(), g.nbox * sizeof(BoxDev), cudaMemcpyHostToDevice,
                      g.stream));
  TRY(cudaStreamSynchronize(g.stream));  // the host records may change again
  ++g.epoch;
  return RT_OK;
}

rt_status rt_set_density(rt_grid_t h, const double* d_nH) { return set_field(h, d_nH, true); }
rt_status rt_set_xHI(rt_grid_t h, const double* d_xHI) { return set_field(h, d_xHI, false); }

rt_status rt_set_sources(rt_grid_t h, int nsrc, const int32_t* d_pos, const int32_t* d_box,
                         const double* d_ndot, const double* d_radius) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_sources: null grid");
  if (nsrc < 0 || nsrc > (1 << 26)) return fail(RT_ERR_INVALID, "rt_set_sources: bad source count");
  if (nsrc > 0 && (!d_pos || !d_ndot || !d_radius))
    return fail(RT_ERR_INVALID, "rt_set_sources: null source array");
  Grid& g = *reinterpret_cast<Grid*>(h);
  ++g.epoch;  // the source arrays, tables and geometry may move
  rt_status st = ingest_sources(g, nsrc, d_pos, d_box, d_ndot, d_radius);
  if (st == RT_OK) {
    const int mmax = std::max(1, std::min(isqrt_h(g.max_r2), g.nmax / 2 + 1));
    st = ensure_geometry(g, mmax);
  }
  if (st == RT_OK) st = ensure_row_tables(g);
  if (st != RT_OK) {  // no kernel may use sources whose geometry or tables are missing
    g.nsrc = 0;
    g.nsrc_in = 0;
    g.max_r2 = 0;
    g.source_voxels = 0;
    g.r2_sorted_h.clear();
  }
  return st;
}

rt_status rt_raytrace(rt_grid_t h, double* d_gamma, int schedule) {
  if (!h) return fail(RT_ERR_INVALID, "rt_raytrace: null grid");
  if (!d_gamma) return fail(RT_ERR_INVALID, "rt_raytrace: null output");
  if (schedule != RT_SCHED_AUTO && schedule != RT_SCHED_PLAIN && schedule != RT_SCHED_BATCHED &&
      schedule != RT_SCHED_BATCHED_EXIT)
    return fail(RT_ERR_INVALID, "rt_raytrace: unknown schedule");
  Grid& g = *reinterpret_cast<Grid*>(h);
  rt_status st = check_ready(g, "rt_raytrace");
  if (st != RT_OK) return st;
  if (schedule == RT_SCHED_AUTO) schedule = g.auto_plain ? RT_SCHED_PLAIN : RT_SCHED_BATCHED;
  TRY(cudaEventRecord(g.ev[0], g.stream));
  const bool rates = schedule != RT_SCHED_PLAIN &&
                     takes_rates_kernels(g, schedule == RT_SCHED_BATCHED_EXIT);
  if (rates && g.interp_mode == RT_INTERP_OPTICAL_DEPTH && !g.od_captured)
    g.od_captured = in_capture(g.stream);
  TRY(launch_precompute(g, rates ? PRE_THICK : PRE_INVN, d_gamma));
  TRY(cudaEventRecord(g.ev[1], g.stream));
  if (g.nsrc > 0) {
    if (schedule == RT_SCHED_PLAIN)
      st = run_trace(g, d_gamma, nullptr, nullptr, g.nsrc, RT_SCHED_PLAIN, g.nsrc);
    else
      st = run_trace(g, d_gamma, nullptr, g.items, 24 * g.nsrc, RT_SCHED_BATCHED, g.nsrc, nullptr,
                     schedule == RT_SCHED_BATCHED_EXIT);
    if (st != RT_OK) return st;
  } else {
    g.stats.launches = 0;
    g.stats.items = 0;
  }
  TRY(cudaEventRecord(g.ev[2], g.stream));
  g.stats.source_voxels = g.source_voxels;
  return RT_OK;
}

rt_status rt_raytrace_source_coldens(rt_grid_t h, int src, double* d_coldens, int schedule) {
  if (!h) return fail(RT_ERR_INVALID, "rt_raytrace_source_coldens: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  if (!d_coldens) return fail(RT_ERR_INVALID, "rt_raytrace_source_coldens: null output");
  if (src < 0 || src >= g.nsrc_in)
    return fail(RT_ERR_INVALID, "rt_raytrace_source_coldens: source index out of range");
  rt_status st = check_ready(g, "rt_raytrace_source_coldens");
  if (st != RT_OK) return st;
  TRY(launch_precompute(g, PRE_DTAU, d_coldens));
  const int hmax = face_hcap(g.max_r2, g.nmax);
  if (schedule != RT_SCHED_PLAIN && g.interp_mode == RT_INTERP_GEOMETRIC && g.nmax <= kMaxBox32 &&
      rates_smem_bytes(hmax, few_items_block(hmax)) <= 227 * 1024) {
    // 24 CTAs, their source looked up on the device, with room for the widest one:
    // nothing is asked back
    TraceArgs a = base_args(g);
    a.coldens = d_coldens;
    a.one_src = g.src_of_input + src;
    a.hcap = hmax;
    const int block = few_items_block(hmax);
    TRY(launch_rates(g, a, block, 24, rates_smem_bytes(hmax, block), 1));
    TRY(launch_tau_to_coldens(g, d_coldens));
    g.stats.launches = 1;
    g.stats.block = block & ~kAhead;
    g.stats.grid = 24;
    g.stats.items = 24;
    g.stats.schedule = RT_SCHED_BATCHED;
    return latched_errors(g);
  }
  int p = 0;
  TRY(cudaMemcpyAsync(&p, g.src_of_input + src, sizeof(int), cudaMemcpyDeviceToHost, g.stream));
  TRY(cudaStreamSynchronize(g.stream));
  int hitems[24];
  for (int q = 0; q < 24; ++q) hitems[q] = (p << 5) | q;
  TRY(cudaMemcpyAsync(g.queue + 8, hitems, 24 * sizeof(int), cudaMemcpyHostToDevice, g.stream));
  if (schedule == RT_SCHED_PLAIN) {
    hitems[0] = p;
    TRY(cudaMemcpyAsync(g.queue + 8, hitems, sizeof(int), cudaMemcpyHostToDevice, g.stream));
    st = run_trace(g, nullptr, d_coldens, g.queue + 8, 1, RT_SCHED_PLAIN, 1);
  } else {
    st = run_trace(g, nullptr, d_coldens, g.queue + 8, 24, RT_SCHED_BATCHED, 0, nullptr, false,
                   g.r2_sorted_h[p]);
  }
  if (st != RT_OK) return st;
  TRY(cudaStreamSynchronize(g.stream));  // hitems is a stack buffer
  return latched_errors(g);
}

rt_status rt_get_stats(rt_grid_t h, rt_stats* out) {
  if (!h || !out) return fail(RT_ERR_INVALID, "rt_get_stats: null argument");
  Grid& g = *reinterpret_cast<Grid*>(h);
  TRY(cudaStreamSynchronize(g.stream));
  float ms = 0.f;
  if (cudaEventElapsedTime(&ms, g.ev[1], g.ev[2]) == cudaSuccess) g.stats.trace_ms = ms;
  if (cudaEventElapsedTime(&ms, g.ev[0], g.ev[1]) == cudaSuccess) g.stats.prep_ms = ms;
  cudaGetLastError();
  unsigned long long rc = 0;
  TRY(cudaMemcpy(&rc, g.counters, sizeof(rc), cudaMemcpyDeviceToHost));
  g.stats.rate_cells = (int64_t)rc;
  g.stats.kernel_launches = g_launches.load();
  g.stats.row_table_bytes = g.rtab ? g.rtab_bytes + g.itab_bytes + g.ftab_bytes : 0;
  *out = g.stats;
  return latched_errors(g);
}

rt_status rt_check(rt_grid_t h) {
  if (!h) return fail(RT_ERR_INVALID, "rt_check: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  return latched_errors(g);
}

rt_status rt_inject_device_error(rt_grid_t h, int bits) {
  if (!h) return fail(RT_ERR_INVALID, "rt_inject_device_error: null grid");
  if (bits <= 0 || bits > (ERR_LAYER_CAP | ERR_GEO | ERR_INPUT | ERR_CUBE))
    return fail(RT_ERR_INVALID, "rt_inject_device_error: unknown error bits");
  Grid& g = *reinterpret_cast<Grid*>(h);
  int cur = 0;
  TRY(cudaStreamSynchronize(g.stream));
  TRY(cudaMemcpy(&cur, g.err, sizeof(int), cudaMemcpyDeviceToHost));
  cur |= bits;
  TRY(cudaMemcpy(g.err, &cur, sizeof(int), cudaMemcpyHostToDevice));
  return RT_OK;
}

rt_status rt_set_device_memory_limit(int64_t bytes) {
  if (bytes < 0) return fail(RT_ERR_INVALID, "rt_set_device_memory_limit: negative limit");
  std::lock_guard<std::mutex> lk(g_mem_mutex);
  mem_limit_locked();  // the environment's value is replaced, not read later
  g_mem_limit = bytes;
  return RT_OK;
}

int64_t rt_device_memory_in_use(void) {
  std::lock_guard<std::mutex> lk(g_mem_mutex);
  return g_mem_live;
}

rt_status rt_chemistry_step(rt_grid_t h, const double* d_gamma, const double* d_x0,
                            const double* d_xavg_in, double dt_s, double alpha_H, double C_H,
                            double conv_tol, double* d_xavg_out, double* d_xnew_out,
                            int64_t* d_unconverged) {
  if (!h) return fail(RT_ERR_INVALID, "rt_chemistry_step: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  if (!d_gamma || !d_x0 || !d_xavg_in || !d_xavg_out || !d_xnew_out || !d_unconverged)
    return fail(RT_ERR_INVALID, "rt_chemistry_step: null pointer");
  if (!(dt_s > 0) || !std::isfinite(dt_s) || !(alpha_H >= 0) || !(C_H >= 0) || !(conv_tol >= 0))
    return fail(RT_ERR_INVALID, "rt_chemistry_step: need dt > 0, alpha_H >= 0, C_H >= 0");
  if (!g.nH) return fail(RT_ERR_STATE, "rt_chemistry_step: rt_set_density not called");
  TRY(launch_chemistry(g, d_gamma, d_x0, d_xavg_in, dt_s, alpha_H, C_H, 1e-10, 50, conv_tol,
                       d_xavg_out, d_xnew_out, d_unconverged, nullptr));
  return RT_OK;
}

rt_status rt_iterate(rt_grid_t h, double* d_x, double dt_s, double alpha_H, double C_H,
                     int max_iter, double conv_tol, double conv_frac, int use_graph,
                     double* d_gamma, int* h_iters) {
  if (!h) return fail(RT_ERR_INVALID, "rt_iterate: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  if (!d_x || !d_gamma) return fail(RT_ERR_INVALID, "rt_iterate: null pointer");
  if (max_iter < 1 || max_iter > 1000 || !(dt_s > 0) || !(alpha_H >= 0) || !(C_H >= 0) ||
      !(conv_tol >= 0) || !(conv_frac >= 0))
    return fail(RT_ERR_INVALID, "rt_iterate: bad arguments");
  if (!g.have_tables) return fail(RT_ERR_STATE, "rt_iterate: rt_set_tables not called");
  if (!g.nH) return fail(RT_ERR_STATE, "rt_iterate: rt_set_density not called");
  const size_t bytes = g.ncell * sizeof(double);
  for (double** p : {&g.xbuf, &g.xavg, &g.xavg2, &g.xhi_int})  // (a call may have got only some)
    if (!*p) TRY(grid_malloc(g, p, bytes));
  g.xHI = g.xhi_int;
  const int64_t limit = (int64_t)std::ceil(conv_frac * (double)g.ncell);
  cudaStream_t user = g.stream;
  if (g.od_scratch && !g.od_captured) g.od_captured = in_capture(user);
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  rt_status st = RT_OK;
  int iters = 0;
  auto body = [&](int k) -> rt_status {
    const int* skip = g.flags;
    double* xin = (k % 2 == 0) ? g.xavg : g.xavg2;
    double* xout = (k % 2 == 0) ? g.xavg2 : g.xavg;
    TRY(launch_one_minus(xin, g.xhi_int, g.ncell, skip, g.stream));
    TRY(launch_precompute(g, takes_rates_kernels(g, false) ? PRE_THICK : PRE_INVN, d_gamma, skip));
    TRY(cudaMemsetAsync(g.unconv, 0, sizeof(int64_t), g.stream));
    if (g.nsrc > 0) {
      rt_status s2 = run_trace(g, d_gamma, nullptr, g.items, 24 * g.nsrc, RT_SCHED_BATCHED, g.nsrc, skip);
      if (s2 != RT_OK) return s2;
    }
    TRY(launch_chemistry(g, d_gamma, d_x, xin, dt_s, alpha_H, C_H, 1e-10, 50, conv_tol, xout,
                         g.xbuf, g.unconv, skip));
    TRY(launch_conv_check(g.unconv, limit, g.flags, g.stream));
    return RT_OK;
  };
  TRY(cudaMemcpyAsync(g.xavg, d_x, bytes, cudaMemcpyDeviceToDevice, user));
  TRY(cudaMemsetAsync(g.flags, 0, 2 * sizeof(int), user));
  if (use_graph) {
    // capture once on a private stream; replay while the arguments and the grid's
    // state are those it was captured with
    const Grid::IterKey key{d_x, d_gamma, dt_s, alpha_H, C_H, conv_tol, conv_frac, max_iter,
                            g.epoch, user};
    if (!g.it_stream) TRY(cudaStreamCreateWithFlags(&g.it_stream, cudaStreamNonBlocking));
    cudaStream_t cap = g.it_stream;
    if (!g.it_exec || !(key == g.it_key)) {
      if (g.it_exec) {
        TRY(cudaStreamSynchronize(cap));  // the old graph may still run
        cudaGraphExecDestroy(g.it_exec);
        g.it_exec = nullptr;
      }
      g.stream = cap;
      g.capturing = true;
      cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        for (int k = 0; k < max_iter && st == RT_OK; ++k) st = body(k);
        cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
        if (st == RT_OK && e2 != cudaSuccess) st = cuda_fail(e2, "cudaStreamEndCapture");
      } else {
        st = cuda_fail(e, "cudaStreamBeginCapture");
      }
      g.capturing = false;
      g.stream = user;
      if (st == RT_OK) {
        cudaError_t e3 = cudaGraphInstantiate(&exec, graph, 0);
        if (e3 != cudaSuccess) st = cuda_fail(e3, "cudaGraphInstantiate");
      }
      if (graph) cudaGraphDestroy(graph);
      if (st != RT_OK) {
        if (exec) cudaGraphExecDestroy(exec);
        return st;
      }
      g.it_exec = exec;
      g.it_key = key;
    }
    cudaError_t e4 = cudaEventRecord(g.ev[3], user);
    if (e4 == cudaSuccess) e4 = cudaStreamWaitEvent(cap, g.ev[3], 0);
    if (e4 == cudaSuccess) e4 = cudaGraphLaunch(g.it_exec, cap);
    if (e4 == cudaSuccess) e4 = cudaEventRecord(g.ev[3], cap);
    if (e4 == cudaSuccess) e4 = cudaStreamWaitEvent(user, g.ev[3], 0);
    if (e4 != cudaSuccess) return cuda_fail(e4, "graph launch");
  } else {
    for (int k = 0; k < max_iter; ++k) {
      st = body(k);
      if (st != RT_OK) return st;
      int fl[2] = {0, 0};
      TRY(cudaMemcpyAsync(fl, g.flags, 2 * sizeof(int), cudaMemcpyDeviceToHost, user));
      TRY(cudaStreamSynchronize(user));
      if (fl[0]) break;
    }
  }
  TRY(cudaMemcpyAsync(d_x, g.xbuf, bytes, cudaMemcpyDeviceToDevice, user));
  if (h_iters) {
    TRY(cudaMemcpyAsync(g.pin + 2, g.flags, 2 * sizeof(int), cudaMemcpyDeviceToHost, user));
    const rt_status err = latched_errors(g);  // (synchronises)
    *h_iters = iters = g.pin[3];
    return err;
  }
  return RT_OK;
}

rt_status rt_raytrace_backward(rt_grid_t h, const double* d_dL_dgamma, double* d_dL_dlog_nHI,
                               double* d_dL_dlog_ndot) {
  if (!h) return fail(RT_ERR_INVALID, "rt_raytrace_backward: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  if (!d_dL_dgamma || !d_dL_dlog_nHI)
    return fail(RT_ERR_INVALID, "rt_raytrace_backward: null pointer");
  if (g.nsrc_in > 0 && !d_dL_dlog_ndot)
    return fail(RT_ERR_INVALID, "rt_raytrace_backward: null dL/dlog Ndot output");
  rt_status st = check_ready(g, "rt_raytrace_backward");
  if (st != RT_OK) return st;
  if (g.interp_mode != RT_INTERP_GEOMETRIC)
    return fail(RT_ERR_INVALID, "rt_raytrace_backward: the adjoint is built for the geometric "
                                "weights (rt_set_interpolation mode 0)");
  TRY(launch_precompute(g, PRE_INVN, d_dL_dlog_nHI));
  if (g.nsrc == 0) return RT_OK;
  if (g.dq_cap < g.nsrc) {
    dev_free(g.dq_merged);
    g.dq_merged = nullptr;
    g.dq_cap = 0;
    TRY(grid_malloc(g, &g.dq_merged, g.nsrc * sizeof(double)));
    g.dq_cap = g.nsrc;
  }
  TRY(cudaMemsetAsync(g.dq_merged, 0, g.nsrc * sizeof(double), g.stream));
  // Whole faces by warps (k_bwd_faces) and quadrants (adjoint_plan).  Quadrant items of large
  // sources by 128-thread CTAs, the rest one per warp (as the trace, but with the warp-mode
  // threshold capped at half-width 27: such a warp keeps two layers and its layer records in
  // shared memory, and beyond 27 too few stay resident -- 1e5 sources of the 250^3 workload
  // took 1.5x longer at 30).
  const int ns = g.nsrc;
  const int* r2s = g.r2_sorted_h.data();
  const int hbig = face_hcap(g.max_r2, g.nmax);
  const int lcap = std::max(1, std::min(isqrt_h(g.max_r2), g.nmax / 2 + 1));
  const bool exit = g.bwd_exit != 0;
  // Few items: the longest face decides (1e3 sources of R = 22, ms: faces 0.99, quadrants
  // 0.51; 4e3 of R = 5..50: 2.18, 2.09; 1e5: 41.8, 55); fewer still, CTAs take every
  // quadrant (64^3, 256 sources: CTAs 0.21, with warps 0.47).
  const bool tables = g.ftab && g.kap_mmax >= 1 && longest_part(g, 6) <= 0.3;
  const int hwarp = !g.explicit_schedule && longest_part(g, 24) > 1.2 ? 0 : std::min(g.hsmall, 27);
  AdjointPlan plan;
  BwdLaunch Lc, Lw, Lf;  // CTAs, warps, faces
  int hw = 0, nfaces = 0;
  size_t stack_c = 0;
  const int hf = std::min(hbig, kBwdFaceHcap);
  auto prepare = [&](bool faces) -> rt_status {  // launches, and memory for them
    plan = adjoint_plan(ns, g.nmax, faces, exit, hbig, kBwdFaceHcap, hwarp,
                        [&](int h) { return first_fitting(g, r2s, ns, h); });
    Lc = Lw = Lf = BwdLaunch();
    Lc.exit = Lw.exit = Lf.exit = exit;
    Lc.lcap = Lw.lcap = lcap;
    if (plan.split > 0) {
      Lc.block = 128;
      Lc.smem = bwd_smem_bytes(hbig, lcap);
      if (Lc.smem > 227 * 1024)
        return fail(RT_ERR_INVALID, "rt_raytrace_backward: radius too large for the shared-memory layers");
      Lc.stack_cap = face_stack_cap(g.max_r2, g.nmax);
      const int maxg = bwd_max_grid(Lc.smem, 128);
      if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace_backward: no occupancy");
      Lc.grid = std::max(1, std::min(24 * plan.split, maxg));
    }
    hw = plan.split < plan.quads ? face_hcap(r2s[plan.split], g.nmax) : 0;
    if (plan.split < plan.quads) {
      Lw.block = 32;
      Lw.smem = bwd_smem_bytes(hw, lcap) * 8;
      Lw.stack_cap = face_stack_cap(r2s[plan.split], g.nmax);
      const int maxg = bwd_max_grid(Lw.smem, 32);
      if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace_backward: no occupancy (warp mode)");
      Lw.grid = std::max(1, std::min((24 * (plan.quads - plan.split) + 7) / 8, maxg));
    }
    nfaces = 6 * (ns - plan.face_begin);
    if (nfaces > 0) {
      Lf.block = 4;
      Lf.stack_cap = (size_t)std::max(g.face_stack, 1);
      int maxg = 0;
      Lf.wpb = 1;
      for (int cand = 8; cand >= 1; --cand) {
        const int mg = bwd_max_grid(bwd_face_smem_bytes(hf) * cand, 4, cand);
        if (mg * cand > maxg * Lf.wpb) {
          maxg = mg;
          Lf.wpb = cand;
        }
      }
      if (maxg <= 0) return fail(RT_ERR_CUDA, "rt_raytrace_backward: no occupancy (faces)");
      Lf.smem = bwd_face_smem_bytes(hf) * Lf.wpb;
      Lf.grid = std::max(1, std::min((nfaces + Lf.wpb - 1) / Lf.wpb, maxg));
      Lf.redo_cap = plan.leftover ? 24 * ns : 0;
      Lf.split_src = plan.split;
    }
    stack_c = Lc.stack_cap * Lc.grid;
    const size_t stack_w = Lw.stack_cap * Lw.grid * 8;
    const size_t stack_f = Lf.stack_cap * Lf.grid * Lf.wpb;  // (before the others, in their place)
    const size_t need = std::max(stack_c + stack_w, stack_f) * sizeof(double2);
    if (need > g.bwd_stack_bytes) {
      dev_free(g.bwd_stack);
      g.bwd_stack = nullptr;
      g.bwd_stack_bytes = 0;
      TRY(grid_malloc(g, &g.bwd_stack, need));
      g.bwd_stack_bytes = need;
    }
    const size_t redo = 2 * (size_t)Lf.redo_cap;
    if (redo > g.bwd_redo_cap) {
      dev_free(g.bwd_redo);
      g.bwd_redo = nullptr;
      g.bwd_redo_cap = 0;
      TRY(grid_malloc(g, &g.bwd_redo, redo * sizeof(int)));
      g.bwd_redo_cap = redo;
    }
    return RT_OK;
  };
  st = prepare(tables);
  // The faces' list takes 192 bytes a source, which the quadrant kernels do without.
  if (st == RT_ERR_OOM && nfaces > 0) st = prepare(false);
  if (st != RT_OK) return st;
  const int face_begin = plan.face_begin, quads = plan.quads, split = plan.split;
  const bool leftover = plan.leftover;
  TraceArgs a = base_args(g);
  a.items = g.items;
  // queue: [0] CTAs, [1] warps, [2] faces, [4], [5] items left over for the first two
  TRY(cudaMemsetAsync(g.queue, 0, 6 * sizeof(int), g.stream));
  TRY(cudaEventRecord(g.ev[1], g.stream));
  g.stats.launches = 0;
  auto launch = [&](BwdLaunch& L, int hcap, int begin, int end, int* queue, double2* stack) {
    TraceArgs b = a;
    b.hcap = hcap;
    b.item_begin = begin;
    b.n_items = end;
    b.queue = queue;
    if (L.n_dev) b.items = L.redo;
    g.stats.launches += 1;
    return launch_trace_bwd(g, b, L, d_dL_dgamma, d_dL_dlog_nHI, g.dq_merged, stack);
  };
  if (nfaces > 0) {
    Lf.redo = g.bwd_redo;
    Lf.redo_n = g.queue + 4;
    TRY(launch(Lf, hf, 6 * face_begin, 6 * ns, g.queue + 2, g.bwd_stack));
  }
  if (leftover) {
    Lc.redo = g.bwd_redo;
    Lc.n_dev = g.queue + 4;
    Lw.redo = g.bwd_redo + Lf.redo_cap;
    Lw.n_dev = g.queue + 5;
  }
  if (split > 0) TRY(launch(Lc, hbig, 0, 24 * split, g.queue, g.bwd_stack));
  if (split < quads)
    TRY(launch(Lw, hw, leftover ? 0 : 24 * split, 24 * quads, g.queue + 1, g.bwd_stack + stack_c));
  TRY(cudaEventRecord(g.ev[2], g.stream));
  TRY(launch_dndot_inputs(g, g.dq_merged, d_dL_dlog_ndot));
  g.stats.block = nfaces > 0 ? 32 * Lf.wpb : split > 0 ? 128 : 32;
  g.stats.grid = nfaces > 0 ? Lf.grid : split > 0 ? Lc.grid : Lw.grid;
  g.stats.items = 24 * ns;
  return RT_OK;
}

rt_status rt_set_interpolation(rt_grid_t h, int mode, double tau_weight_min) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_interpolation: null grid");
  if (mode != RT_INTERP_GEOMETRIC && mode != RT_INTERP_OPTICAL_DEPTH)
    return fail(RT_ERR_INVALID, "rt_set_interpolation: unknown mode");
  if (!(tau_weight_min > 0.0) || !std::isfinite(tau_weight_min))
    return fail(RT_ERR_INVALID, "rt_set_interpolation: tau_weight_min must be finite and > 0");
  Grid& g = *reinterpret_cast<Grid*>(h);
  if (mode == RT_INTERP_OPTICAL_DEPTH && !g.od_scratch) {
    // Room for the reciprocals of every resident warp of rates.cu: no more than their layers
    // take of the SMs' shared memory.  Here once, so that a trace allocates nothing and may
    // be captured; where it fails, trace.cu, which needs none.  Kept when the mode goes back
    // (a caller's graph may hold it), but given up where the grid needs the memory
    // (release_scratch).  A capture under way, on whatever stream, is none of this call's
    // business: relaxed mode lets the allocation through without ending it.
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool clear = cudaPeekAtLastError() == cudaSuccess;
    cudaStreamCaptureMode relaxed = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&relaxed);
    const cudaError_t e = dev_malloc(&g.od_scratch, (size_t)sms * 228 * 1024);
    cudaThreadExchangeStreamCaptureMode(&relaxed);
    if (e != cudaSuccess && clear) cudaGetLastError();  // (an error that was there stays)
  }
  g.interp_mode = mode;
  g.tau_w0 = tau_weight_min;
  ++g.epoch;
  return RT_OK;
}

rt_status rt_set_adjoint_mode(rt_grid_t h, int stop_at_opaque) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_adjoint_mode: null grid");
  reinterpret_cast<Grid*>(h)->bwd_exit = stop_at_opaque ? 1 : 0;
  return RT_OK;
}

rt_status rt_set_schedule(rt_grid_t h, int block_big, int hsmall, int hface) {
  if (!h) return fail(RT_ERR_INVALID, "rt_set_schedule: null grid");
  if (block_big != 128 && block_big != 256)
    return fail(RT_ERR_INVALID, "rt_set_schedule: block must be 128 or 256");
  if (hsmall < 0 || hsmall > 32)
    return fail(RT_ERR_INVALID, "rt_set_schedule: hsmall must be 0..32");
  if (hface < 0 || hface > 20)
    return fail(RT_ERR_INVALID, "rt_set_schedule: hface must be 0..20");
  Grid& g = *reinterpret_cast<Grid*>(h);
  g.block_big = block_big;
  g.hsmall = hsmall;
  g.hface = hface;
  g.explicit_schedule = true;
  ++g.epoch;
  return RT_OK;
}

// Key of a workload for the autotuner cache: box sizes and the distribution of
// traced radii (what the schedule's performance depends on).
static std::string tune_key(const Grid& g) {
  std::vector<int> r2 = g.r2_sorted_h;  // descending
  auto pct = [&](double q) { return r2.empty() ? 0 : r2[(size_t)((1.0 - q) * (r2.size() - 1))]; };
  std::ostringstream k;
  k << "nbox=" << g.nbox << ",nmax=" << g.nmax << ",ncell=" << g.ncell << ",nsrc=" << g.nsrc
    << ",r2max=" << g.max_r2 << ",r2p50=" << pct(0.5) << ",r2p90=" << pct(0.9);
  return k.str();
}

rt_status rt_autotune(rt_grid_t h, const char* cache_path, int* h_block, int* h_hsmall,
                      int* h_hface) {
  if (!h) return fail(RT_ERR_INVALID, "rt_autotune: null grid");
  Grid& g = *reinterpret_cast<Grid*>(h);
  ++g.epoch;  // the schedule may change
  rt_status st = check_ready(g, "rt_autotune");
  if (st != RT_OK) return st;
  auto report = [&]() {
    if (h_block) *h_block = g.block_big;
    if (h_hsmall) *h_hsmall = g.hsmall;
    if (h_hface) *h_hface = g.hface;
  };
  const std::string key = tune_key(g);
  if (cache_path) {
    std::ifstream in(cache_path);
    std::string line;
    while (std::getline(in, line)) {
      std::istringstream ls(line);
      std::string k;
      int b = 0, hs = -1, hf = -1, ap = -1;
      std::string how;
      if ((ls >> k >> b >> hs >> hf >> ap) && k == key && (b == 128 || b == 256) && hs >= 0 &&
          hs <= 32 && hf >= 0 && hf <= 20 && (ap == 0 || ap == 1)) {
        g.block_big = b;
        g.hsmall = hs;
        g.hface = hf;
        g.auto_plain = ap;
        g.explicit_schedule = !((ls >> how) && how == "rule");
        report();
        return RT_OK;
      }
    }
  }
  if (g.nsrc == 0) {
    report();
    return RT_OK;
  }
  double* gam = nullptr;
  TRY(grid_malloc(g, &gam, g.ncell * sizeof(double)));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // time of one batched trace in the current configuration (second of two runs)
  auto timed = [&](float& t) {
    for (int rep = 0; rep < 2 && st == RT_OK; ++rep) {
      cudaEventRecord(e0, g.stream);
      st = rt_raytrace(h, gam, RT_SCHED_BATCHED);
      cudaEventRecord(e1, g.stream);
      cudaEventSynchronize(e1);
      cudaEventElapsedTime(&t, e0, e1);
    }
    return st == RT_OK;
  };
  // stage 1: CTA size x warp-mode threshold (whole-face warps off); stage 2: the
  // whole-face threshold at the chosen pair
  const int blocks[] = {128, 256};
  const int hss[] = {0, 11, 15, 19, 22, 24, 27, 30};
  const int hfs[] = {9, 11, 13, 15, 17, 19};
  // stage 0: the rule on sizes (rates.cu's kernels only), kept unless thresholds beat it
  float best = 1e30f, rule = 1e30f;
  int bb = g.block_big, bh = g.hsmall, bf = 0;
  const bool was_explicit = g.explicit_schedule;
  g.explicit_schedule = false;
  if (takes_rates_kernels(g, false)) timed(rule);
  g.explicit_schedule = true;
  g.hface = 0;
  for (int b : blocks)
    for (int hs : hss) {
      if (st != RT_OK) break;
      g.block_big = b;
      g.hsmall = hs;
      float t = 0.f;
      if (!timed(t)) break;
      if (t < best) {
        best = t;
        bb = b;
        bh = hs;
      }
    }
  g.block_big = bb;
  g.hsmall = bh;
  for (int hf : hfs) {
    if (st != RT_OK || bh == 0) break;
    g.hface = hf;
    float t = 0.f;
    if (!timed(t)) break;
    if (t < best) {
      best = t;
      bf = hf;
    }
  }
  // stage 2b: the warp-mode threshold again, with the chosen whole-face threshold
  // (whole faces take the small sources away from the warp mode, which shifts its
  // best range)
  if (bf > 0) {
    g.hface = bf;
    for (int hs : hss) {
      if (st != RT_OK) break;
      if (hs == 0 || hs == bh) continue;
      g.hsmall = hs;
      float t = 0.f;
      if (!timed(t)) break;
      if (t < best) {
        best = t;
        bh = hs;
      }
    }
    g.hsmall = bh;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  dev_free(gam);
  if (st != RT_OK) {
    g.explicit_schedule = was_explicit;
    return st;
  }
  g.hface = bf;
  if (rule <= best) {  // reported as the closest thresholds
    best = rule;
    g.explicit_schedule = false;
    g.block_big = bb = 128;
    g.hsmall = bh = 32;
    g.hface = bf = 16;
  }
  // stage 3: the paper's block-per-source schedule against the tuned batched one
  // (RT_SCHED_AUTO then takes the faster)
  if (st == RT_OK) {
    float tp = 0.f;
    TRY(grid_malloc(g, &gam, g.ncell * sizeof(double)));
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, g.stream);
    st = rt_raytrace(h, gam, RT_SCHED_PLAIN);
    cudaEventRecord(e1, g.stream);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(&tp, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    dev_free(gam);
    if (st != RT_OK) return st;
    g.auto_plain = tp < best ? 1 : 0;
  }
  report();
  if (cache_path) {
    std::ofstream out(cache_path, std::ios::app);
    out << key << " " << bb << " " << bh << " " << bf << " " << g.auto_plain
        << (g.explicit_schedule ? "" : " rule") << "\n";
  }
  return RT_OK;
}

void rt_grid_destroy(rt_grid_t h) {
  if (!h) return;
  Grid* g = reinterpret_cast<Grid*>(h);
  cudaStreamSynchronize(g->stream);
  free_grid(g);
}

}  // extern "C"
