// K1: fine propagator F (Sec. 3.1) -- implicit Euler steps of eq. (fd), batched over
// independent states (time slices and requests), on register tiles of thread-block clusters
// (fine_tile.cuh).  This file holds the host side: layouts and launch plans.
//
// Per implicit step  (I - dtau R_h) u^{m+1} = u^m  the increment  d = u^{m+1} - u^m  solves
//   (I - dtau R_h) d = dtau R_h w,   w = u^m inside, g(tau^{m+1}) on the far edges,
// with d = 0 on the far edges.  It is solved by Jacobi sweeps
//   d <- (b + sum_k c_k d_k) / (1 + sum_k c_k + r dtau),   b = dtau R_h w,
// started from zero in the first step of a call, from the previous increment in the second and from
// the extrapolation of the previous two after that.  The Gershgorin bound q < 1 of the system
// (checked on the host) makes every sweep a max-norm contraction by q; the sweep count is
// chosen so that q^sweeps is below a target (2^-22, 2^-10, 2^-6 up to step 15 and 1/2 from there)
// and extrapolated starts converge (capi.cu: extrap_stable).  The state is a compensated
// pair (hi, lo): u = hi + lo, updated by an error-free two-sum, so that increments below half
// an ulp of u are not lost over tens of thousands of steps; b is evaluated from hi.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fine_tile.cuh"

namespace bsp {

// u_out = hi + lo from the second workspace half (after a single launch over several regions,
// which may not write u_out: it may alias u_in, and regions read their neighbours' nodes)
__global__ void fine_finish_kernel(const __grid_constant__ FineBatch fb) {
  const ItemDesc& d = fb.it[blockIdx.y];
  const size_t MM = (size_t)fb.M * fb.M;
  const float* ws = fb.ws + (size_t)blockIdx.y * 8 * MM;
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e < MM) d.out[e] = ws[4 * MM + e] + ws[5 * MM + e];
}

// A layout: tiles of tc columns x tr rows per lane, clusters of C CTAs, ntx x nty regions that
// overlap so that a launch may run H sweeps (one region: any number).
struct FineLayout {
  int tc, tr, C, ntx, nty, H;
};

#define BS_FINE_DISPATCH(tc, tr, CALL)                 \
  switch ((tc) * 10 + (tr)) {                          \
    case 24: return CALL(2, 4);                        \
    case 44: return CALL(4, 4);                        \
    case 64: return CALL(6, 4);                        \
    case 84: return CALL(8, 4);                        \
    case 22: return CALL(2, 2);                        \
    case 42: return CALL(4, 2);                        \
    case 62: return CALL(6, 2);                        \
    case 82: return CALL(8, 2);                        \
  }

static int layout_launch(const FineLayout& y, const FineBatch& fb, const FineLaunch& fl, bool spread, cudaStream_t s) {
#define CALL(TC, TR) fine_tile_launch<TC, TR>(fb, fl, spread, s)
  BS_FINE_DISPATCH(y.tc, y.tr, CALL)
#undef CALL
  return set_error(BS_ERR_ARG, "fine propagator: no tile of %d x %d", y.tc, y.tr);
}

static int layout_capacity(const FineLayout& y) {
#define CALL(TC, TR) fine_tile_capacity<TC, TR>(y.C)
  BS_FINE_DISPATCH(y.tc, y.tr, CALL)
#undef CALL
  return 0;
}

// Sweeps that n regions of w nodes on an m-node axis leave exact: each region loses that many
// nodes at a cut edge, and together they cover the axis.  A multiple of 4, so that the parts that
// are written start at multiples of 4 where the regions do.
static int axis_overlap(int n, int w, int m) {
  int h = 1 << 30;
  for (int t = 0; t + 1 < n; ++t) h = std::min(h, (w - region_origin(t + 1, n, w, m) + region_origin(t, n, w, m)) / 2);
  return h & ~3;
}

static FineLayout make_layout(int M, int tc, int tr, int C, int hmin) {
  FineLayout y = {tc, tr, C, 1, 1, 0};
  const int w = 32 * tc, r = C * kFineWarps * tr;
  auto regions = [&](int len) {
    if (M <= len) return 1;
    for (int n = 2;; ++n)
      if (axis_overlap(n, len, M) >= hmin) return n;
  };
  y.ntx = regions(w);
  y.nty = regions(r);
  y.H = std::min(axis_overlap(y.ntx, w, M), axis_overlap(y.nty, r, M));
  return y;
}

// Estimated time of a late (two-sweep) step of nb states, in SM clocks: waves of clusters times
// the clocks of a CTA's step (fitted to 2.4k to 6.5k clocks measured for 1024 to 8192 nodes per
// CTA) and, over several regions, a launch's load, setup and store (about 27k clocks at 8192
// nodes) per step.  A layout without a known capacity (clusters above 8 CTAs may not fit the device)
// comes after every layout with one.
static double layout_cost(const FineLayout& y, int nb) {
  const int cap = layout_capacity(y);
  const double clusters = (double)nb * y.ntx * y.nty;
  const double waves = cap > 0 ? std::ceil(clusters / cap) : 1e9 * clusters * y.C;
  const double nodes = 32.0 * y.tc * kFineWarps * y.tr;
  double t = 1800.0 + 0.57 * nodes;
  if (y.ntx * y.nty > 1) t += (3000.0 + 1.3 * nodes) / std::max(1, std::min(y.H, 1 << 10) / 2);
  return waves * t;
}

// Columns per lane of a region that is as wide as the grid (M <= 256).
static int tile_columns(int M) { return 2 * ((M + 63) / 64); }

// The layout of a launch batch of nb states: the one with the least estimated time.  For M <= 256
// that is 32-row CTAs for a batch and 16-row CTAs, twice as many per state, while they fit the
// GPU (one 256 x 256 state, per step: 1.81 us against 3.15; 64 states 17.6 against 15.3).  Over
// several regions, 1024 x 1024 takes 256 x 288 nodes (30 states, per step: 172 us against 184
// for 256 x 256).  BS_OPT_FINE_TILE forces one: 1 is 32-row CTAs (beyond
// one cluster, regions of 256 x 256), 2 is 16-row CTAs (beyond one cluster, regions of 256 x 288).
static FineLayout choose_layout(int M, int nb) {
  if (M <= 256) {
    const int tc = tile_columns(M);
    const FineLayout y4 = make_layout(M, tc, 4, (M + 31) / 32, 1), y2 = make_layout(M, tc, 2, (M + 15) / 16, 1);
    if (g_opt.fine_tile == 1 || g_opt.fine_tile == 2) return g_opt.fine_tile == 2 ? y2 : y4;
    return layout_cost(y2, nb) < layout_cost(y4, nb) ? y2 : y4;
  }
  constexpr int kMinOverlap = 12;
  if (g_opt.fine_tile == 1) return make_layout(M, 8, 4, 8, kMinOverlap);
  if (g_opt.fine_tile == 2) return make_layout(M, 8, 4, 9, kMinOverlap);
  FineLayout best = {};
  double best_cost = 1e300;
  for (int tc = 4; tc <= 8; tc += 4)
    for (int C = 4; C <= 9; ++C) {
      const FineLayout y = make_layout(M, tc, 4, C, kMinOverlap);
      const double c = layout_cost(y, nb);
      if (c < best_cost) {
        best_cost = c;
        best = y;
      }
    }
  return best;
}

// The largest sweep count of any item in step `step`.
static int max_step_sweeps(const ItemDesc* items, int n, int step) {
  int m = 1;
  for (int k = 0; k < n; ++k) m = std::max(m, step_sweeps(items[k], step));
  return m;
}

// Launch plan over several regions: whole steps are packed into a launch while their sweeps
// (the largest count of any item, step by step) add up to at most hmax; a step with more sweeps
// than that is split evenly over several launches.
static void fine_plan(const ItemDesc* items, int n, int nsteps, int hmax, std::vector<FineLaunch>& plan) {
  plan.clear();
  int step = 0;
  while (step < nsteps) {
    const int m = max_step_sweeps(items, n, step);
    if (m > hmax) {
      const int nl = (m + hmax - 1) / hmax;
      const int chunk = (m + nl - 1) / nl;
      for (int s0 = 0; s0 < m; s0 += chunk) plan.push_back({step, 1, s0, std::min(m, s0 + chunk), 0, 0, 0});
      ++step;
      continue;
    }
    int h = m, k = 1;
    while (step + k < nsteps) {
      const int mk = max_step_sweeps(items, n, step + k);
      if (h + mk > hmax) break;
      h += mk;
      ++k;
    }
    plan.push_back({step, k, 0, 1 << 30, 0, 0, 0});
    step += k;
  }
  for (size_t l = 0; l < plan.size(); ++l) {
    plan[l].first = l == 0;
    plan[l].last = l + 1 == plan.size() && l > 0;
    plan[l].par = (int)(l & 1);
  }
}

int fine_launches(const bs_grid* g, const ItemDesc* items, int n, int nsteps) {
  if (nsteps < 1) return 0;
  const FineLayout y = choose_layout(g->M, std::min(n, kMaxItems));
  if (y.ntx * y.nty == 1) return (n + kMaxItems - 1) / kMaxItems;
  int total = 0;
  std::vector<FineLaunch> plan;
  for (int base = 0; base < n; base += kMaxItems) {
    fine_plan(items + base, std::min(n - base, kMaxItems), nsteps, y.H, plan);
    total += (int)plan.size() + (plan.size() == 1 ? 1 : 0);
  }
  return total;
}

int fine_cluster_ctas(const bs_grid* g) { return g->M <= 256 ? (g->M + 31) / 32 : 0; }

int fine_cluster_capacity(const bs_grid* g) {
  if (g->M > 256) return 0;
  return layout_capacity(make_layout(g->M, tile_columns(g->M), 4, (g->M + 31) / 32, 1));
}

static int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      v = 0;
    }
    return v;
  }();
  return n;
}

int launch_fine(const bs_grid* g, const ItemDesc* items, int n, int nsteps, cudaStream_t s) {
  if (nsteps < 1) return BS_OK;
  const int M = g->M;
  const size_t MM = (size_t)M * M;
  const FineLayout y = choose_layout(M, std::min(n, kMaxItems));
  const bool single = y.ntx * y.nty == 1;
  FineBatch fb;
  fb.ws = nullptr;
  if (!single) {
    int rc = ensure(const_cast<bs_grid*>(g)->ws_fine, (size_t)std::min(n, kMaxItems) * 8 * MM * sizeof(float));
    if (rc) return rc;
    fb.ws = (float*)g->ws_fine.ptr;
  }
  fb.status = g->status;
  fb.M = M;
  fb.C = y.C;
  fb.ntx = y.ntx;
  fb.nty = y.nty;
  fb.H = y.H;
  fb.h = (float)(g->xmax / (M - 1));
  std::vector<FineLaunch> plan;
  for (int base = 0; base < n; base += kMaxItems) {
    fb.n = std::min(n - base, kMaxItems);
    for (int k = 0; k < fb.n; ++k) fb.it[k] = items[base + k];
    const bool spread = fb.n * y.C * y.ntx * y.nty <= sm_count();
    int rc;
    if (single) {
      // one cluster holds the state: every step in one launch, in place if u_out aliases u_in
      if ((rc = layout_launch(y, fb, {0, nsteps, 0, 1 << 30, 1, 1, 0}, spread, s))) return rc;
      continue;
    }
    fine_plan(fb.it, fb.n, nsteps, y.H, plan);
    for (const FineLaunch& fl : plan)
      if ((rc = layout_launch(y, fb, fl, spread, s))) return rc;
    if (plan.size() == 1) {
      fine_finish_kernel<<<dim3((unsigned)((MM + 255) / 256), fb.n), 256, 0, s>>>(fb);
      BS_CUDA_TRY(cudaGetLastError());
    }
  }
  return BS_OK;
}

}  // namespace bsp
