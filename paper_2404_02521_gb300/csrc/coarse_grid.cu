// Numerical coarse propagator G and the serial Parareal sweep on grids beyond one cluster's shared
// memory (M > 256): the solver of coarse.cu (BiCGSTAB on the Jacobi-scaled system, right
// preconditioned with M^{-1} = 2I - A^, extrapolated first guesses) with its vectors in a global
// workspace, one cooperative launch per call.
//
// A state is owned by a group of blocks, one tile of kCgW x kCgH nodes per block or several (cg_layout).
// Where a state may get more or fewer blocks, its sums are kept per tile and added in the tiles'
// order; every rounding is explicit, so its result does not depend on how many it got.  An iteration
// is two passes over the group's tiles, each followed by one barrier of the group that also carries
// its dot products:
//   A  x += omega M^{-1} s, r = s - omega t, p = r + beta (p - omega v), v = A^ M^{-1} p:
//      (r^, v), (r, r)
//   B  x += alpha M^{-1} p, s = r - alpha v, t = A^ M^{-1} s: (t, s), (t, t), (r^, s), (r^, t)
// A pass stages its operand (p or s) in shared memory with two halo rows and columns, forming it
// from the vectors that its owners wrote before the last barrier, evaluates M^{-1} of it on the
// tile and one halo row and column, and then the product; nothing is exchanged in between.
// p and v alternate between two buffers, because a neighbour may still read the old ones.
//
// What bounds it: two barriers, two rounds of L2 loads and the latency of short passes per
// iteration, 10.6 us at 512 x 512 on 128 blocks (49.5 us in the former layout, one cluster of 16
// SMs with eight cluster barriers and every vector update through L2).  64 x 32 tiles keep a
// 512 x 512 state's vectors in the registers of one block per tile (12% of the staged nodes
// are halo); up to 304 tiles are resident, above that (about 770 x 770) a block passes its
// tiles through the workspace (1024 x 1024: 25.4 us per iteration, 172 on one cluster).  States of a
// batched launch run side by side in groups of blocks, then one after another (10 states of
// 301 x 301: 2.5 us per iteration and state, 7.0 on clusters).
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "grid_barrier.cuh"

namespace bsp {

constexpr int kCgThreads = 256;
constexpr int kCgW = 64, kCgH = 32;                 // nodes of a tile
constexpr int kCgK = kCgW * kCgH / kCgThreads;      // nodes of a thread: a strip of one column
constexpr int kCgS = kCgW + 4;                      // row length of the staged operands: two halo columns
constexpr int kCgHalo = 2 * 2 * kCgS + 2 * 2 * kCgH;          // nodes of an operand's halo
constexpr int kCgRing = 2 * (kCgW + 2) + 2 * kCgH;            // nodes of its inner ring
constexpr int kCgAttempts = 3;                      // BiCGSTAB starts per implicit step
constexpr int kCgVectors = 13;
constexpr int kCgArrivalStride = 32;                // a cache line per group's counter

struct CgArgs {
  ItemDesc d;        // dtau = coarse step
  SweepArgs a;
  float* ws;         // per group: kCgVectors vectors of M*M
  float4* partials;  // per group: [2][tiles], the tiles' sums
  double2* npart;    // [2][group_blocks]: norms of a sweep (one group)
  unsigned* arrivals;   // per group, kCgArrivalStride apart, zero at launch
  int M, tiles, group_blocks, groups;
  float h;
};

// Every multiply-add of this file is explicit and it is compiled without implicit contraction: a ring
// node of M^{-1} p equals its owner's bit for bit, and a state's result is the same whether its tiles
// stay in registers or not.

// row_coefs with the drift fused in
__device__ __forceinline__ void cg_row(const ItemDesc& d, int j, float& cs, float& cn, float& gj) {
  gj = (float)j;
  const float b = d.ay * (gj * gj);
  cs = fmaf(d.my, gj, b);
  cn = fmaf(-d.my, gj, b);
}

// weighted neighbours of a node
__device__ __forceinline__ float cg_off(float nW, float nC, float nE, float cW, float cE, float sW, float sC, float sE,
                                        float ce, float cw, float cs, float cn, float cg) {
  float t = ce * cE;
  t = fmaf(cw, cW, t);
  t = fmaf(cs, sC, t);
  t = fmaf(cn, nC, t);
  return fmaf(cg, (sE - nE) - (sW - nW), t);
}

// ONE: every block owns one tile, whose Krylov vectors stay in registers; only the nodes that a
// neighbour stages (two rows and columns along the tile's edges) are written to the workspace.
// Otherwise a pass loads and stores them tile by tile.  PER_SM: blocks that share an SM.  A block that
// has an SM to itself adds the sums of its tiles in registers, others keep them per tile (TILE_SUMS).
template <bool ONE, int PER_SM>
__global__ void __launch_bounds__(kCgThreads, PER_SM) sweep_grid_kernel(const __grid_constant__ CgArgs ca) {
  constexpr int K = kCgK;
  constexpr bool TILE_SUMS = PER_SM > 1;
  const ItemDesc& d = ca.d;
  const SweepArgs& a = ca.a;
  const int M = ca.M, tid = threadIdx.x;
  const size_t MM = (size_t)M * M;
  const int group = blockIdx.x / ca.group_blocks;
  GridGroup<kCgThreads> grid{ca.arrivals + group * kCgArrivalStride, ca.partials + (size_t)group * 2 * ca.tiles, ca.tiles, a.status,
                             (int)blockIdx.x % ca.group_blocks, ca.group_blocks, tid};
  float* w0 = ca.ws + (size_t)group * kCgVectors * MM;
  float *const gu = w0, *const gx = w0 + MM, *const gxp = w0 + 2 * MM, *const gxq = w0 + 3 * MM, *const gr = w0 + 4 * MM,
              *const grh = w0 + 5 * MM, *const gs = w0 + 6 * MM, *const gt = w0 + 7 * MM, *const gq = w0 + 8 * MM;
  float* const gp[2] = {w0 + 9 * MM, w0 + 10 * MM};
  float* const gv[2] = {w0 + 11 * MM, w0 + 12 * MM};
  __shared__ float P[kCgS * (kCgH + 4)], Q[kCgS * (kCgH + 4)];
  const PayoffF pf = make_payoff(d);
  const float rdt = d.rdt, tol = (float)a.tol;
  const int tiles_i = (M + kCgW - 1) / kCgW, tiles = ca.tiles;
  const int tc = tid % kCgW, r0 = tid / kCgW * K;   // the thread's column and first row of a tile
  const int L0 = (r0 + 2) * kCgS + tc + 2;          // and its index in P and Q
  int i0 = 0, j0 = 0;
  float ce = 0.f, cw = 0.f, cgi = 0.f, id[K];       // of the current tile's strip; id is 0 off the PDE rows

  auto enter = [&](int tile) {
    j0 = tile / tiles_i * kCgH;
    i0 = tile % tiles_i * kCgW;
    const int i = i0 + tc;
    column_coefs(d, i, ce, cw, cgi);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int j = j0 + r0 + k;
      id[k] = i < M - 1 && j < M - 1 ? inv_diag(d, i, j) : 0.f;
    }
  };
  auto each_tile = [&](auto&& body) {
    if constexpr (ONE) {
      body(grid.block);
    } else {
      for (int tile = grid.block; tile < tiles; tile += grid.blocks) {
        enter(tile);
        body(tile);
        __syncthreads();   // the staged operands are rewritten
        if (TILE_SUMS) grid.flush();
      }
    }
  };
  auto reduce4 = [&](float (&v)[4]) {
    if (TILE_SUMS) grid.total(v, tiles);
    else grid.sum(v);
  };
  if constexpr (ONE) enter(grid.block);
  // f(k, e) for the nodes of the strip that lie in the grid, e their index
  auto strip = [&](auto&& f) {
    const int i = i0 + tc;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int j = j0 + r0 + k;
      if (i < M && j < M) f(k, (size_t)j * M + i);
    }
  };
  auto load = [&](const float* g, float (&v)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.f;
    strip([&](int k, size_t e) { v[k] = g[e]; });
  };
  auto store = [&](float* g, const float (&v)[K]) { strip([&](int k, size_t e) { g[e] = v[k]; }); };
  // what a neighbour stages (ONE) or the next pass loads
  auto share = [&](float* g, const float (&v)[K]) {
    strip([&](int k, size_t e) {
      if (!ONE || tc < 2 || tc >= kCgW - 2 || r0 + k < 2 || r0 + k >= kCgH - 2) g[e] = v[k];
    });
  };
  auto advance = [](float (&y)[K], float a, const float (&d)[K]) {   // y += a d
#pragma unroll
    for (int k = 0; k < K; ++k) y[k] = fmaf(a, d[k], y[k]);
  };
  // own nodes of an operand into its tile
  auto put = [&](float* dst, const float (&v)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) dst[L0 + k * kCgS] = v[k];
  };
  // its halo: val(e) inside the grid, zero outside
  auto halo = [&](float* dst, auto&& val) {
#pragma unroll
    for (int n = 0; n < (kCgHalo + kCgThreads - 1) / kCgThreads; ++n) {
      const int h = tid + n * kCgThreads;
      if (h >= kCgHalo) break;
      int row, c;
      if (h < 4 * kCgS) {
        const int w = h / kCgS;
        row = w < 2 ? w : w + kCgH;
        c = h - w * kCgS;
      } else {
        const int w = h - 4 * kCgS;
        row = 2 + (w >> 2);
        c = (w & 1) + ((w & 2) ? kCgW + 2 : 0);
      }
      const int i = i0 + c - 2, j = j0 + row - 2;
      dst[row * kCgS + c] = i >= 0 && i < M && j >= 0 && j < M ? val((size_t)j * M + i) : 0.f;
    }
  };
  // f(k, y, A^ y) down the strip, y the operand's nodes
  auto product = [&](const float* src, auto&& f) {
    const float* y = src + L0;
    float nW = y[-kCgS - 1], nC = y[-kCgS], nE = y[-kCgS + 1], cW = y[-1], cC = y[0], cE = y[1];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float sW = y[(k + 1) * kCgS - 1], sC = y[(k + 1) * kCgS], sE = y[(k + 1) * kCgS + 1];
      float cs, cn, gj;
      cg_row(d, j0 + r0 + k, cs, cn, gj);
      f(k, cC, fmaf(-id[k], cg_off(nW, nC, nE, cW, cE, sW, sC, sE, ce, cw, cs, cn, cgi * gj), cC));
      nW = cW; nC = cC; nE = cE;
      cW = sW; cC = sC; cE = sE;
    }
  };
  // Q = M^{-1} P = 2 P - A^ P on the tile (also in q) and one ring around it, then av = A^ Q
  auto precond_product = [&](float (&q)[K], float (&av)[K]) {
    __syncthreads();
    product(P, [&](int k, float y, float ay) {
      q[k] = fmaf(2.f, y, -ay);
      Q[L0 + k * kCgS] = q[k];
    });
    if (tid < kCgRing) {
      int row, c;
      if (tid < 2 * (kCgW + 2)) {
        row = tid < kCgW + 2 ? 1 : kCgH + 2;
        c = 1 + (tid < kCgW + 2 ? tid : tid - (kCgW + 2));
      } else {
        const int w = tid - 2 * (kCgW + 2);
        row = 2 + (w >> 1);
        c = (w & 1) ? kCgW + 2 : 1;
      }
      const int i = i0 + c - 2, j = j0 + row - 2;
      float val = 0.f;
      if (i >= 0 && i < M - 1 && j >= 0 && j < M - 1) {
        float e, w, g, cs, cn, gj;
        column_coefs(d, i, e, w, g);
        cg_row(d, j, cs, cn, gj);
        const float* y = P + row * kCgS + c;
        val = fmaf(2.f, y[0], -fmaf(-inv_diag(d, i, j),
                                    cg_off(y[-kCgS - 1], y[-kCgS], y[-kCgS + 1], y[-1], y[1], y[kCgS - 1], y[kCgS],
                                           y[kCgS + 1], e, w, cs, cn, g * gj),
                                    y[0]));
      }
      Q[row * kCgS + c] = val;
    }
    __syncthreads();
    product(Q, [&](int k, float, float aq) { av[k] = aq; });
  };

  const bool batched = a.mode == SWEEP_PROP && a.nprop > 0;
  const int nstates = batched ? a.nprop : 1;
  const int n_lo = a.n_end > 0 ? a.n_begin : a.n_first;
  const int n_hi = a.n_end > 0 ? a.n_end : (a.mode == SWEEP_PROP ? a.n_first + 1 : a.N);
  int iters_max = 0, iters_total = 0, nsolves = 0;
  bool failed = false;
  // the strip's x, r (s after an iteration's first pass), r^, p, v, t and M^{-1} p (then M^{-1} s)
  float x[K], r[K], rh[K], p[K], v[K], t[K], q[K];
  // of a tile in the workspace: where a block has its SM's registers, its loads are all in flight at once
  // and its stores come last; else x is done with before the others are loaded
  constexpr bool EARLY = PER_SM == 1;
  auto advance_x = [&](float a) {
    advance(x, a, q);
    store(gx, x);
  };

  for (int st = group; st < nstates && !grid.dead; st += ca.groups) {
    const PropItem pit = batched ? a.prop[st] : PropItem{a.in, a.out, d.tau0};
    const float* src = a.mode == SWEEP_PROP   ? pit.in
                       : a.mode == SWEEP_INIT ? a.U + (size_t)n_lo * MM
                       : n_lo == a.n_first    ? a.Gold + (size_t)a.n_first * MM   // G(u_k) unchanged: G_old_k
                                              : a.U + (size_t)n_lo * MM;
    each_tile([&](int) {
      strip([&](int, size_t e) {
        gu[e] = src[e];
        gx[e] = 0.f;
        gxp[e] = 0.f;
        gxq[e] = 0.f;
      });
    });
    int nhist = 0;
    for (int n = n_lo; n < n_hi && !grid.dead; ++n) {
      const bool skip_g = a.mode == SWEEP_ITER && n == a.n_first;
      for (int cstep = 0; cstep < (skip_g ? 0 : a.csteps) && !grid.dead; ++cstep) {
        const float tau_new = (float)(pit.tau0 + a.slice_len * n + (cstep + 1) * d.dtau);
        // far-field data, and the first guess 3 d_{m-1} - 3 d_{m-2} + d_{m-3} (gx holds d_{m-1})
        each_tile([&](int) {
          strip([&](int k, size_t e) {
            const int i = i0 + tc, j = j0 + r0 + k;
            if (i == M - 1 || j == M - 1) gu[e] = far_field(pf, i * ca.h, j * ca.h, tau_new);
            const float d1 = gx[e], d2 = gxp[e];
            if (nhist >= 3) gx[e] = fmaf(3.f, d1 - d2, gxq[e]);
            else if (nhist == 2) gx[e] = fmaf(2.f, d1, -d2);
            gxq[e] = d2;
            gxp[e] = d1;
          });
        });
        int it = 0;
        bool conv = false, fail = true;
        // a breakdown (a zero denominator) restarts from the current iterate
        for (int attempt = 0; attempt < kCgAttempts && !conv && fail && !grid.dead; ++attempt) {
          grid.barrier();   // the owners' u and x are visible
          // b^ = D^{-1} dtau R_h u;  r = r^ = p = b^ - A^ x
          float sums[4] = {0.f, 0.f, 0.f, 0.f};
          each_tile([&](int tile) {
            if (TILE_SUMS) sums[0] = sums[1] = sums[2] = sums[3] = 0.f;
            load(gx, x);
            float u[K], ax[K];
            load(gu, u);
            put(P, u);
            put(Q, x);
            halo(P, [&](size_t e) { return __ldcg(gu + e); });
            halo(Q, [&](size_t e) { return __ldcg(gx + e); });
            __syncthreads();
            product(Q, [&](int k, float, float ay) { ax[k] = ay; });
            const float* y = P + L0;
#pragma unroll
            for (int k = 0; k < K; ++k, y += kCgS) {
              float cs, cn, gj;
              cg_row(d, j0 + r0 + k, cs, cn, gj);
              const float c = y[0];
              float b = ce * (y[1] - c);
              b = fmaf(-cw, c - y[-1], b);
              b = fmaf(cs, y[kCgS] - c, b);
              b = fmaf(-cn, c - y[-kCgS], b);
              b = fmaf(cgi * gj, (y[kCgS + 1] - y[-kCgS + 1]) - (y[kCgS - 1] - y[-kCgS - 1]), b);
              b = fmaf(-rdt, c, b);
              const float bh = b * id[k];
              r[k] = rh[k] = p[k] = bh - ax[k];
              sums[0] = fmaf(bh, bh, sums[0]);
              sums[1] = fmaf(r[k], r[k], sums[1]);
            }
            share(gr, r);
            share(gp[0], p);
            if (!ONE) store(grh, rh);
            if (TILE_SUMS) grid.put(sums, tile);
          });
          reduce4(sums);
          float rho = sums[1];
          const float stop2 = tol * tol * sums[0];
          conv = sums[1] <= stop2 || !(sums[0] > 1e-30f);
          fail = false;
          float alpha = 0.f, omega = 0.f, beta = 0.f;
          bool open = false;   // the last iteration's x += omega M^{-1} s is still to be applied
          for (int m = 0; !conv && !fail && it < a.maxit && !grid.dead; ++m) {
            ++it;
            const float *vo = gv[m ? (m - 1) & 1 : 0], *po = gp[m ? (m - 1) & 1 : 0];
            float *vn = gv[m & 1], *pn = gp[m & 1];
            float sa[4] = {0.f, 0.f, 0.f, 0.f};
            each_tile([&](int tile) {
              if (TILE_SUMS) sa[0] = sa[1] = sa[2] = sa[3] = 0.f;
              if (!ONE) {
                if (EARLY) load(grh, rh);
                load(po, p);
                if (m == 0) {
                  load(gr, r);
                } else {
                  load(gx, x);
                  load(gq, q);
                  if (!EARLY) advance_x(omega);
                  load(gs, r);
                  load(gt, t);
                  load(vo, v);
                }
              }
              if (m == 0) {   // r and p are at hand
                halo(P, [&](size_t e) { return __ldcg(po + e); });
              } else {
                halo(P, [&](size_t e) {
                  const float rr = fmaf(-omega, __ldcg(gt + e), __ldcg(gs + e));
                  return fmaf(beta, fmaf(-omega, __ldcg(vo + e), __ldcg(po + e)), rr);
                });
                if (ONE || EARLY) advance(x, omega, q);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                  r[k] = fmaf(-omega, t[k], r[k]);
                  p[k] = fmaf(beta, fmaf(-omega, v[k], p[k]), r[k]);
                }
                share(gr, r);
                share(pn, p);
              }
              put(P, p);
              precond_product(q, v);
              if (!ONE && !EARLY) {
                store(gq, q);
                load(grh, rh);
              }
#pragma unroll
              for (int k = 0; k < K; ++k) {
                sa[0] = fmaf(rh[k], v[k], sa[0]);
                sa[1] = fmaf(r[k], r[k], sa[1]);
              }
              share(vn, v);
              if (!ONE && EARLY) {
                store(gq, q);
                if (m) store(gx, x);
              }
              if (TILE_SUMS) grid.put(sa, tile);
            });
            open = false;
            reduce4(sa);
            if (sa[1] <= stop2) {
              conv = true;
              break;
            }
            if (sa[0] == 0.f) {
              fail = true;
              break;
            }
            alpha = rho / sa[0];
            float sb[4] = {0.f, 0.f, 0.f, 0.f};
            each_tile([&](int tile) {
              if (TILE_SUMS) sb[0] = sb[1] = sb[2] = sb[3] = 0.f;
              if (!ONE) {
                if (EARLY) load(grh, rh);
                load(gx, x);
                load(gq, q);
                if (!EARLY) advance_x(alpha);
                load(gr, r);
                load(vn, v);
              }
              halo(P, [&](size_t e) { return fmaf(-alpha, __ldcg(vn + e), __ldcg(gr + e)); });
              if (ONE || EARLY) advance(x, alpha, q);
              advance(r, -alpha, v);
              share(gs, r);
              put(P, r);
              precond_product(q, t);
              if (!ONE && !EARLY) {
                store(gq, q);
                load(grh, rh);
              }
#pragma unroll
              for (int k = 0; k < K; ++k) {
                sb[0] = fmaf(t[k], r[k], sb[0]);
                sb[1] = fmaf(t[k], t[k], sb[1]);
                sb[2] = fmaf(rh[k], r[k], sb[2]);
                sb[3] = fmaf(rh[k], t[k], sb[3]);
              }
              share(gt, t);
              if (!ONE && EARLY) {
                store(gq, q);
                store(gx, x);
              }
              if (TILE_SUMS) grid.put(sb, tile);
            });
            reduce4(sb);
            open = true;
            omega = sb[1] > 0.f ? sb[0] / sb[1] : 0.f;
            const float rho_new = fmaf(-omega, sb[3], sb[2]);
            if (omega == 0.f || rho == 0.f) {
              fail = true;
              beta = 0.f;
            } else {
              beta = (rho_new / rho) * (alpha / omega);
              rho = rho_new;
            }
          }
          each_tile([&](int) {
            if (!ONE) {
              load(gx, x);
              load(gq, q);
            }
            if (open) advance(x, omega, q);
            store(gx, x);
          });
        }
        if (!conv) failed = true;
        iters_max = max(iters_max, it);
        iters_total += it;
        ++nsolves;
        nhist = nhist < 3 ? nhist + 1 : 3;
        each_tile([&](int) { strip([&](int, size_t e) { gu[e] += gx[e]; }); });
      }
      if (a.mode == SWEEP_PROP) {
        each_tile([&](int) { strip([&](int, size_t e) { pit.out[e] = gu[e]; }); });
        continue;
      }
      // correction u_{n+1} = F_n + (G_new - G_old_n), squares in FP32 (u_new - u_old of nearby
      // values is exact), sums in FP64
      double n0 = 0.0, n1 = 0.0;
      float* Un = a.U + (size_t)(n + 1) * MM;
      const float* Fn = a.Fb + (size_t)n * MM;
      float* Gn = a.Gold + (size_t)n * MM;
      each_tile([&](int) {
        strip([&](int, size_t e) {
          const float gnew = gu[e];
          if (a.mode == SWEEP_INIT) {
            Un[e] = gnew;
            Gn[e] = gnew;
            n0 += (double)(gnew * gnew);
          } else {
            const float unew = Fn[e] + (gnew - Gn[e]), du = unew - Un[e];
            Un[e] = unew;
            Gn[e] = gnew;
            gu[e] = unew;
            n0 += (double)(unew * unew);
            n1 += (double)(du * du);
          }
        });
      });
      __shared__ double2 wn[kCgThreads / 32];
      auto reduce = [&](double& b0, double& b1) {   // over the block, the same in all threads
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          b0 += __shfl_xor_sync(0xffffffffu, b0, off);
          b1 += __shfl_xor_sync(0xffffffffu, b1, off);
        }
        __syncthreads();
        if ((tid & 31) == 0) wn[tid >> 5] = make_double2(b0, b1);
        __syncthreads();
        b0 = b1 = 0.0;
        for (int w = 0; w < kCgThreads / 32; ++w) {
          b0 += wn[w].x;
          b1 += wn[w].y;
        }
      };
      reduce(n0, n1);
      double2* np = ca.npart + (n & 1) * ca.group_blocks;
      if (tid == 0) __stcg(np + grid.block, make_double2(n0, n1));
      grid.barrier();
      if (grid.block == 0) {   // (the slots alternate by slice: the next slice's barriers order their reuse)
        n0 = n1 = 0.0;
        for (int b = tid; b < grid.blocks; b += kCgThreads) {
          const double2 w = __ldcg(np + b);
          n0 += w.x;
          n1 += w.y;
        }
        reduce(n0, n1);
        if (tid == 0) {
          a.norms[2 * (n + 1)] = n0;
          a.norms[2 * (n + 1) + 1] = a.mode == SWEEP_ITER ? n1 : 0.0;
        }
      }
    }
    if (batched && st + ca.groups < nstates) grid.barrier();   // the next state reuses the vectors
  }
  if (grid.block == 0 && tid == 0) {
    if (failed && !grid.dead) atomicOr(a.status, 1);
    atomicMax(a.status + 1, iters_max);
    atomicAdd(a.status + 2, iters_total);
    atomicAdd(a.status + 3, nsolves);
    if (a.mode == SWEEP_ITER && n_hi == a.N) {
      double num = 0.0, den = 0.0;
      for (int n = 1; n <= a.N; ++n) {
        den = fmax(den, a.norms[2 * n]);
        if (n >= a.n_first + 1) num = fmax(num, a.norms[2 * n + 1]);
      }
      a.defect[0] = den > 0.0 ? sqrt(num) / sqrt(den) : sqrt(num);
    }
  }
}

// Blocks of the solver that the current device runs at once, measured once per device.
template <bool ONE, int PER_SM>
static int cg_blocks(int* out) {
  static std::mutex mu;
  static int known[64] = {};
  int dev = 0;
  BS_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  int n = dev < 64 ? known[dev] : 0;
  if (!n) {
    int per_sm = 0, sms = 0;
    BS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sweep_grid_kernel<ONE, PER_SM>, kCgThreads, 0));
    BS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    n = std::min(per_sm * sms, kGridMaxBlocks);
    if (n < 1) return set_error(BS_ERR_CUDA, "coarse propagator: no block of the grid solver fits an SM");
    if (dev < 64) known[dev] = n;
  }
  *out = n;
  return BS_OK;
}

// Layout of a launch of nst states.
//  - Up to as many tiles as blocks are resident (about 770 nodes per axis): the layout with the least
//    estimated time, rounds of states times microseconds per iteration.  A tile per block takes 12; with the
//    tiles through the workspace it is 1 and 11.5 for every tile of a block, a quarter more where the
//    groups' vectors exceed the L2 (fitted to 11.8 to 62 us at 512 to 700 nodes, one to eight groups).  A
//    state that needs more than half of the resident blocks would leave the rest idle and the next
//    states waiting: 7 states of 520 x 520, 2 steps, 12.0 ms in one group of 153 blocks and 6.9 in
//    seven of 43; 64 of 512 x 512 56 and 49 ms.
//  - Up to three tiles per SM, a block per SM: 22.8 us per iteration at 800 x 800, 25.1 with two.
//  - Beyond, two blocks per SM (1024 x 1024: 25.4 us, 28.8 with one), in the groups with the least
//    estimated time (8 states 65 and 49 ms).
// The sums are added in the same order within each of the three ranges, so a state's result does not
// depend on the others of its launch.
enum CgKind { CG_ONE, CG_SHARED, CG_ALONE };   // a tile per block; several, two blocks or one block per SM
struct CgLayout {
  CgKind kind;
  int group_blocks, groups;
};
static CgLayout cg_layout(int M, int tiles, int nst, const int (&blocks)[3]) {   // blocks: resident, by kind
  constexpr int kMaxGroups = 8;
  constexpr double kOneUs = 12.0, kPassUs = 1.0, kTileUs = 11.5, kL2Bytes = 110e6, kBeyondL2 = 1.25;
  if (tiles > blocks[CG_ONE] && tiles <= 3 * blocks[CG_ALONE]) return {CG_ALONE, std::min(tiles, blocks[CG_ALONE]), 1};
  auto rounds = [&](int groups) { return (double)((nst + groups - 1) / groups); };
  CgLayout best = {};
  double cost = 1e300;
  if (tiles <= blocks[CG_ONE]) {
    best = {CG_ONE, tiles, std::min(nst, blocks[CG_ONE] / tiles)};
    cost = 0.97 * rounds(best.groups) * kOneUs;   // the others have to gain something
  }
  for (int g = 1; g <= std::min({nst, kMaxGroups, blocks[CG_SHARED]}); ++g) {
    const int gb = std::min(tiles, blocks[CG_SHARED] / g);
    double us = kPassUs + kTileUs * ((tiles + gb - 1) / gb);
    if (g > 1 && 4.0 * kCgVectors * g * M * M > kL2Bytes) us *= kBeyondL2;
    if (rounds(g) * us < cost) {
      cost = rounds(g) * us;
      best = {CG_SHARED, gb, g};
    }
  }
  return best;
}

int launch_sweep_grid(const bs_grid* g, const ItemDesc& d, const SweepArgs& a, cudaStream_t s) {
  const int M = g->M;
  const size_t MM = (size_t)M * M;
  const int nst = a.mode == SWEEP_PROP && a.nprop > 0 ? a.nprop : 1;
  const int tiles = ((M + kCgW - 1) / kCgW) * ((M + kCgH - 1) / kCgH);
  int blocks[3] = {}, rc;
  if ((rc = cg_blocks<true, 2>(blocks + CG_ONE)) || (rc = cg_blocks<false, 2>(blocks + CG_SHARED)) ||
      (rc = cg_blocks<false, 1>(blocks + CG_ALONE)))
    return rc;
  const CgLayout y = cg_layout(M, tiles, nst, blocks);
  CgArgs ca;
  ca.tiles = tiles;
  ca.group_blocks = y.group_blocks;
  ca.groups = y.groups;
  // vectors, the tiles' sums, norm partials, arrivals
  const size_t fbytes = ((size_t)ca.groups * kCgVectors * MM * sizeof(float) + 255) & ~(size_t)255;
  const size_t pbytes = (size_t)ca.groups * 2 * tiles * sizeof(float4);
  const size_t nbytes = (size_t)2 * ca.group_blocks * sizeof(double2);
  const size_t abytes = (size_t)ca.groups * kCgArrivalStride * sizeof(unsigned);
  rc = ensure(const_cast<bs_grid*>(g)->ws_coarse, fbytes + pbytes + nbytes + abytes);
  if (rc) return rc;
  unsigned char* ws = static_cast<unsigned char*>(g->ws_coarse.ptr);
  ca.d = d;
  ca.a = a;
  ca.ws = reinterpret_cast<float*>(ws);
  ca.partials = reinterpret_cast<float4*>(ws + fbytes);
  ca.npart = reinterpret_cast<double2*>(ws + fbytes + pbytes);
  ca.arrivals = reinterpret_cast<unsigned*>(ws + fbytes + pbytes + nbytes);
  ca.M = M;
  ca.h = (float)(g->xmax / (M - 1));
  BS_CUDA_TRY(cudaMemsetAsync(ca.arrivals, 0, abytes, s));
  void* args[] = {&ca};
  void* const kernels[] = {reinterpret_cast<void*>(sweep_grid_kernel<true, 2>),
                           reinterpret_cast<void*>(sweep_grid_kernel<false, 2>),
                           reinterpret_cast<void*>(sweep_grid_kernel<false, 1>)};
  void* kern = kernels[y.kind];
  BS_CUDA_TRY(cudaLaunchCooperativeKernel(kern, dim3(ca.group_blocks * ca.groups),
                                          dim3(kCgThreads), args, 0, s));
  return BS_OK;
}

}  // namespace bsp
