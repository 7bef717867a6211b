// K1 device code: register tiles of the fine propagator F (Sec. 3.1, eq. fd + implicit Euler).
//
// One thread-block cluster owns a region of W = 32 TC columns and C x 8 TR rows of one state and
// steps it without touching memory beyond the SMs: CTA `rank` holds 8 TR rows, each of its 8
// warps TR whole rows of the region, each lane a tile of TR x TC nodes.  The state's high word,
// the increment, the right-hand side and the inverse diagonal of a tile live in registers for
// all steps of a launch, the compensation word and the previous increment in shared memory at
// thread-private addresses (an odd number of pairs per lane: conflict-free).
//
// Why this shape.  The stepper is bound by FP32 arithmetic, issue and the latency of the row
// exchange (an implicit step is two 9-point sweeps, the right-hand side and an error-free
// update; HBM carries 32 B per node per launch of many steps).  A strip of one column per
// thread read its west and east neighbours and its own words from shared memory and took a
// block and a cluster barrier per sweep: 94 issued instructions per node-step, 22 of them memory.
// In a tile the columns come in pairs (one packed instruction for two nodes), west and east
// columns move by warp shuffles, and only the tile's first and last rows pass through shared
// memory: 40 issued instructions per node-step.  Measured on a GB300 at 2070 MHz, before and
// after: 64 states of 256 x 256, 512 steps, 14.1 -> 7.6 ms (the packed FP32 pipe 46% busy); one
// such state 2.00 -> 0.88 ms; 8 states of 64 x 64, 256 steps, 0.67 -> 0.28 ms; 32 states of
// 1024 x 1024, 1024 steps, 219 -> 171 ms.  What is left is latency: two warps per scheduler
// leave the FP32 pipe idle while both load, shuffle or wait.
//
// Exchange.  A warp needs one row from the warp above and one from the warp below, each sweep.
// Sweeps run alternately down and up over the tile's rows with one block barrier in their
// middle, so that each edge row is published half a sweep or more before a neighbour reads it.
// Across CTAs the rows go by st.async, which completes its bytes on an mbarrier of the
// receiving warp (312 clocks per exchange on a probe, 595 to 620 with remote stores and a
// cluster barrier; a block barrier 77, local mbarriers 250).  A row is rewritten two sweeps
// later, after its writer has received the neighbour's rows of the sweep between, which
// the neighbour sent after reading it.
//
// Regions.  A grid that fits one region runs all steps in one launch.  Larger grids are covered
// by overlapping regions, the first aligned with the domain's lower edge and the last with its
// far edge; at a cut edge every sweep costs one more row or column of exactness, so a launch's
// sweeps add up to at most the overlap allows, and (hi, lo, increment, previous increment) go
// through a ping-pong workspace between launches.  The far-edge nodes are always the last
// column of lane 31 and the last row of the last warp (a region that is wider than the grid
// starts at a negative index; nodes outside the domain are inert: zero state, zero invd).
//
// Compiled without implicit contraction; every multiply-add is explicit, and each node is
// computed with the same operations from its global indices in every layout, so results do not
// depend on the layout, the batch or the launch plan.
#pragma once

#include "band.cuh"
#include "cluster_async.cuh"

namespace bsp {

// Pairs of FP32 values in a register pair: one instruction operates on both halves, each rounded
// like the scalar operation.  On this GPU the packed forms run at the scalar rate per value (two
// cycles each) but take half the issue slots.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2pack(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float f2lo(f2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2hi(f2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f2 f2add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Asynchronous 4-byte global -> shared copy; with ok == false the destination is zero-filled
// and nothing is read.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
// ... and the 16-byte one (L2 only)
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

constexpr int kFineWarps = 8;
constexpr int kFineThreads = 32 * kFineWarps;

struct FineBatch {
  ItemDesc it[kMaxItems];
  float* ws;         // per item: [2][hi, lo, increment, previous increment][M*M] (several regions)
  int* status;       // bit 1: an exchange timed out
  int n, M, C;
  int ntx, nty, H;   // regions per axis and the overlap a launch consumes
  float h;
};

// One launch: steps [step0, step0 + nstep) of every item, or with nstep == 1 the sweeps
// [s_begin, s_end) of that step (the step is applied if it ends in this launch).  first: the
// state comes from the items' inputs (no increments yet); last: the result goes to the items'
// outputs instead of the workspace; par: the workspace half that is read.
struct FineLaunch {
  int step0, nstep, s_begin, s_end, first, last, par;
};

template <int TC, int TR>
struct FineShape {
  static_assert(TC % 2 == 0, "columns are paired");
  static constexpr int W = 32 * TC, BH = kFineWarps * TR, H = TC / 2;
  static constexpr int HP = H | 1, WP = 32 * HP;    // pairs per lane and per edge row (odd: conflict-free)
  static constexpr int PS = (TR * H) | 1;           // pairs per lane in a thread-private array
  static constexpr int T = 32 / TR;                 // steps per far-field chunk: one value per lane
  static constexpr int SLOTS = 2 * kFineWarps + 2;  // edge rows: halo, (top, bottom) per warp, halo
  // bytes: thread-private compensation words and previous increments; then the increments' edge
  // rows [2 parities], the state's edge rows and the far row [3 chunks][T], which share their
  // space with the four staging planes of the prologue and epilogue; then the far column
  // [warps][2 chunks][32] and the mbarriers [2 parities][from above, from below], far row [3]
  static constexpr size_t LO = 0, DP = LO + (size_t)kFineThreads * PS * 8, DR = DP + (size_t)kFineThreads * PS * 8,
                          HR = DR + 2 * SLOTS * WP * 8, FF = HR + SLOTS * WP * 8, END = FF + 3 * T * WP * 8;
  static constexpr size_t PLANE = (size_t)BH * W, S0 = DR, SEND = S0 + 4 * PLANE * 4;   // floats; bytes
  static constexpr size_t FC = END > SEND ? END : SEND, MB = FC + kFineWarps * 64 * 4, BYTES = MB + 7 * 8;
  static_assert(FC % 16 == 0 && BYTES <= 227 * 1024, "shared memory of a CTA");
};

// First index of region t of n regions of w nodes on an m-node axis: the first region starts at
// 0, the last ends at m - 1 (a single region ends there too); multiples of 4 where m is one, for
// 16-byte copies.
__host__ __device__ __forceinline__ int region_origin(int t, int n, int w, int m) {
  const int o = n == 1 ? m - w : t * (m - w) / (n - 1);
  return n > 1 && m % 4 == 0 && t < n - 1 ? o & ~3 : o;
}

// A lane's tile: pair c of a row holds columns c and c + TC / 2, so that a pair's north and south
// neighbours are pairs of the rows above and below and its west and east neighbours the pairs
// c - 1 and c + 1, except at the two seams of a row.
template <int TC, int TR>
struct FineTileState {
  using L = FineShape<TC, TR>;
  static constexpr int H = L::H, WP = L::WP;
  f2 d[TR][H], b[TR][H], iv[TR][H], hi[TR][H];
  f2 ce[H], cw[H], cgi[H];         // column coefficients
  float cs[TR], cn[TR], gj[TR];    // row coefficients
  float nrdt;
  int lane, warp, rank;
  f2 *lo, *dp;           // this thread's compensation words and previous increments
  f2 *dr, *hr;           // edge-row buffers at this lane
  int wofs, eofs;        // words from there to the west and east neighbours' (the region's ends: own) word
  int nslot, sslot;      // the rows above and below the tile (its own where the region ends)
  uint64_t* mb;          // [2 parities][from above, from below]
  bool edge_n, edge_s;   // the row above / below is another CTA's
  bool dead;             // a wait ran out

  // A row with its neighbours: x[c + 1] pair c, x[0] and x[H + 1] the pairs shifted out at either end.
  struct Row {
    f2 x[H + 2];
  };
  __device__ __forceinline__ static void seams(Row& o, float w, float e) {
    o.x[0] = f2pack(w, f2lo(o.x[H]));
    o.x[H + 1] = f2pack(f2hi(o.x[1]), e);
  }
  // an own row, by shuffles (at the region's ends the own word, whose weight is zero on the
  // domain's edge)
  __device__ __forceinline__ Row own(const f2 (&v)[H]) const {
    Row o;
#pragma unroll
    for (int c = 0; c < H; ++c) o.x[c + 1] = v[c];
    const float w = __shfl_up_sync(0xffffffffu, f2hi(v[H - 1]), 1), e = __shfl_down_sync(0xffffffffu, f2lo(v[0]), 1);
    seams(o, lane == 0 ? f2lo(v[0]) : w, lane == 31 ? f2hi(v[H - 1]) : e);
    return o;
  }
  // a published row
  __device__ __forceinline__ Row fetch(const f2* row) const {
    Row o;
#pragma unroll
    for (int c = 0; c < H; ++c) o.x[c + 1] = row[c];
    const float* w = reinterpret_cast<const float*>(row);
    seams(o, w[wofs], w[eofs]);
    return o;
  }

  // waits for the row that a neighbour CTA sent in publication q (bounded)
  template <bool STATE>
  __device__ __forceinline__ void await(uint32_t q, bool above) {
    uint64_t* m = mb + (q & 1) * 2 + (above ? 0 : 1);
    if (lane == 0) mbar_arm(m, (STATE ? 2 : 1) * L::W * 4);
    if (!dead) dead = !mbar_wait(m, (q >> 1) & 1);
  }
  // publication q of one edge row of the increment, with STATE also of hi: to the CTA's warps,
  // and from the CTA's first or last row to the neighbour CTA's halo slot
  template <bool STATE, bool TOP>
  __device__ __forceinline__ void publish(uint32_t q) {
    constexpr int r = TOP ? 0 : TR - 1;
    f2* base = dr + (int)(q & 1) * L::SLOTS * WP;
    if (TOP ? edge_n : edge_s) {
      const int to = TOP ? rank - 1 : rank + 1, slot = TOP ? L::SLOTS - 1 : 0;
      const uint32_t m = cluster_addr(smem_addr(mb + (q & 1) * 2 + (TOP ? 1 : 0)), to);
      const uint32_t a = cluster_addr(smem_addr(base + slot * WP), to);
#pragma unroll
      for (int c = 0; c < H; ++c) st_async_v2(a + 8 * c, f2lo(d[r][c]), f2hi(d[r][c]), m);
      if (STATE) {
        const uint32_t ah = cluster_addr(smem_addr(hr + slot * WP), to);
#pragma unroll
        for (int c = 0; c < H; ++c) st_async_v2(ah + 8 * c, f2lo(hi[r][c]), f2hi(hi[r][c]), m);
      }
    }
    f2* st = base + (1 + 2 * warp + (TOP ? 0 : 1)) * WP;
#pragma unroll
    for (int c = 0; c < H; ++c) st[c] = d[r][c];
    if (STATE) {
      f2* sh = hr + (1 + 2 * warp + (TOP ? 0 : 1)) * WP;
#pragma unroll
      for (int c = 0; c < H; ++c) sh[c] = hi[r][c];
    }
  }

  // Row r of a sweep from the old increments n, o, s of the rows above, of and below it, and
  // with FIRST the right-hand side b = dtau R_h hi (eq. fd in index units) from the same rows
  // of hi: the four axis neighbours join b in one chain of fused multiply-adds, then the mixed
  // term, then the diagonal scale.  Differences are written so that no operand needs a sign
  // change.
  template <bool FIRST>
  __device__ __forceinline__ void row(int r, const Row& n, const Row& o, const Row& s, const Row& hn, const Row& ho,
                                      const Row& hs) {
    const f2 cs2 = f2pack(cs[r], cs[r]), cn2 = f2pack(cn[r], cn[r]), gj2 = f2pack(gj[r], gj[r]);
    const f2 rd2 = f2pack(nrdt, nrdt);
#pragma unroll
    for (int c = 0; c < H; ++c) {
      const f2 cg = f2mul(cgi[c], gj2);
      if (FIRST) {
        const f2 hc = ho.x[c + 1];
        f2 t = f2mul(ce[c], f2sub(ho.x[c + 2], hc));
        t = f2fma(cw[c], f2sub(ho.x[c], hc), t);
        t = f2fma(cs2, f2sub(hs.x[c + 1], hc), t);
        t = f2fma(cn2, f2sub(hn.x[c + 1], hc), t);
        t = f2fma(cg, f2sub(f2sub(hs.x[c + 2], hn.x[c + 2]), f2sub(hs.x[c], hn.x[c])), t);
        b[r][c] = f2fma(rd2, hc, t);
      }
      f2 t = f2fma(cw[c], o.x[c], b[r][c]);
      t = f2fma(ce[c], o.x[c + 2], t);
      t = f2fma(cs2, s.x[c + 1], t);
      t = f2fma(cn2, n.x[c + 1], t);
      t = f2fma(cg, f2sub(f2sub(s.x[c + 2], n.x[c + 2]), f2sub(s.x[c], n.x[c])), t);
      d[r][c] = f2mul(t, iv[r][c]);
    }
  }

  // Applies the increments of row r to the state (error-free two-sum of (hi, lo) += v, then
  // renormalise) and turns them into the next step's first guess: with EXTRAP the linear
  // extrapolation 2 d_m - d_{m-1}.
  template <bool EXTRAP>
  __device__ __forceinline__ void commit(int r) {
#pragma unroll
    for (int c = 0; c < H; ++c) {
      const f2 v = d[r][c], h0 = hi[r][c], s = f2add(h0, v), bb = f2sub(s, h0);
      const f2 err = f2add(f2sub(h0, f2sub(s, bb)), f2sub(v, bb));
      const f2 l = f2add(lo[r * H + c], err), hn = f2add(s, l);
      lo[r * H + c] = f2sub(l, f2sub(hn, s));
      hi[r][c] = hn;
      const f2 prev = dp[r * H + c];
      dp[r * H + c] = v;
      if (EXTRAP) d[r][c] = f2sub(f2add(v, v), prev);
    }
  }

  // One Jacobi sweep from the rows of publication q; its edge rows are publication q + 1 unless
  // `pub` is off.  COMMIT: 0 none, 1 the step ends here, 2 the same with the extrapolated guess;
  // `far` then moves the far-edge data of a row to the next step.
  //
  // The rows are updated in order, DOWN or upwards, each after the old values of the row before
  // it were kept, so the first edge row is published at the sweep's start and the other at its
  // end.  With MID the block barrier stands between: a sweep in the other direction must
  // follow, which reads the rows this sweep publishes first at its start and the others after
  // its own barrier, so every row has half a sweep to arrive.  Without MID the barrier stands
  // at the sweep's start and sweeps may follow each other in the same direction.
  template <bool FIRST, int COMMIT, bool DOWN, bool MID, class Far>
  __device__ __forceinline__ void sweep(uint32_t q, bool pub, Far far) {
    if (!MID) __syncthreads();
    const f2* rows = dr + (int)(q & 1) * L::SLOTS * WP;
    constexpr int r_in = DOWN ? 0 : TR - 1, step = DOWN ? 1 : -1;
    // the row k of the sweep's order (TR: the row beyond the tile), from registers or memory
    auto get = [&](int k, Row& x, Row& y) {
      const int r = r_in + (k < TR ? k : 0) * step;
      if (k < TR) {
        x = own(d[r]);
        if (FIRST) y = own(hi[r]);
      } else {
        if (DOWN ? edge_s : edge_n) await<FIRST>(q, !DOWN);
        x = fetch(rows + (DOWN ? sslot : nslot) * WP);
        if (FIRST) y = fetch(hr + (DOWN ? sslot : nslot) * WP);
      }
    };
    Row prev, cur, next, after, hprev, hcur, hnext, hafter;
    get(0, cur, hcur);
    if (TR > 2) get(1, next, hnext);
    if (DOWN ? edge_n : edge_s) await<FIRST>(q, DOWN);
    prev = fetch(rows + (DOWN ? nslot : sslot) * WP);
    if (FIRST) hprev = fetch(hr + (DOWN ? nslot : sslot) * WP);
    if (TR <= 2) get(1, next, hnext);
#pragma unroll
    for (int k = 0; k < TR; ++k) {
      const int r = r_in + k * step;
      if (MID && k == TR / 2) __syncthreads();
      // one row ahead where the barrier has been passed
      if (TR > 2 && k + 2 <= TR) get(k + 2, after, hafter);
      if (TR <= 2 && k + 1 == TR) get(TR, next, hnext);
      if (DOWN) row<FIRST>(r, prev, cur, next, hprev, hcur, hnext);
      else row<FIRST>(r, next, cur, prev, hnext, hcur, hprev);
      if (COMMIT) {
        commit<COMMIT == 2>(r);
        far(r);
      }
      if (pub) {
        if (r == 0) publish<COMMIT != 0, true>(q + 1);
        if (r == TR - 1) publish<COMMIT != 0, false>(q + 1);
      }
      prev = cur;
      cur = next;
      if (TR > 2) next = after;
      if (FIRST) {
        hprev = hcur;
        hcur = hnext;
        if (TR > 2) hnext = hafter;
      }
    }
  }
};

// CTAs of an instance that share an SM: small tiles leave registers for more than one.
constexpr int fine_blocks_per_sm(int tc, int tr) { return tc * tr <= 8 ? 2 : 1; }

template <int TC, int TR>
__global__ void __launch_bounds__(kFineThreads, fine_blocks_per_sm(TC, TR)) fine_tile_kernel(const __grid_constant__ FineBatch fb,
                                                                    const FineLaunch fl) {
  using L = FineShape<TC, TR>;
  constexpr int WP = L::WP, T = L::T, H = L::H, W = L::W;
  cg::cluster_group cluster = cg::this_cluster();
  const ItemDesc& d = fb.it[blockIdx.z];
  const int M = fb.M, C = fb.C;
  const size_t MM = (size_t)M * M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = C > 1 ? (int)cluster.block_rank() : 0;
  const int tx = (int)blockIdx.y % fb.ntx, ty = (int)blockIdx.y / fb.ntx;
  const int R = C * L::BH;
  const int ix0 = region_origin(tx, fb.ntx, L::W, M), jy0 = region_origin(ty, fb.nty, R, M);
  const int row0 = jy0 + rank * L::BH + warp * TR;   // the warp's first row
  const int col0 = ix0 + lane * TC;                  // the lane's first column
  const PayoffF pf = make_payoff(d);

  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t* mb = reinterpret_cast<uint64_t*>(smem + L::MB);
  uint64_t* far_mb = mb + 4;
  FineTileState<TC, TR> s;
  s.lane = lane;
  s.warp = warp;
  s.rank = rank;
  s.lo = reinterpret_cast<f2*>(smem + L::LO) + threadIdx.x * L::PS;
  s.dp = reinterpret_cast<f2*>(smem + L::DP) + threadIdx.x * L::PS;
  s.dr = reinterpret_cast<f2*>(smem + L::DR) + lane * L::HP;
  s.hr = reinterpret_cast<f2*>(smem + L::HR) + lane * L::HP;
  s.wofs = lane == 0 ? 0 : 2 * (H - 1 - L::HP) + 1;   // the west lane's last column: high half of its last pair
  s.eofs = lane == 31 ? 2 * (H - 1) + 1 : 2 * L::HP;
  s.mb = mb;
  s.edge_n = warp == 0 && rank > 0;
  s.edge_s = warp == kFineWarps - 1 && rank < C - 1;
  s.nslot = rank > 0 || warp > 0 ? 2 * warp : 1 + 2 * warp;
  s.sslot = rank < C - 1 || warp < kFineWarps - 1 ? 2 * warp + 3 : 2 * warp + 2;
  s.dead = false;
  s.nrdt = -d.rdt;
  if (threadIdx.x == 0) {
    for (int k = 0; k < 7; ++k) mbar_init(mb + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }

  // The warp's own rows of (hi, lo, increment, previous increment) arrive in four staging planes by
  // asynchronous copies, coalesced along the row, all in flight at once; nodes outside the
  // domain are zero.  16-byte copies where the grid and the input allow them (a chunk then lies
  // wholly inside or outside), else 4-byte ones.  A copy that only fills zeros names the plane's
  // own array: the source has to be aligned to the copy even where nothing is read.  Chunks of four columns are swizzled, so that
  // a lane reads its columns of a row as whole chunks without bank conflicts.
  auto plane_at = [](int r, int c) { return r * W + (((c >> 2) ^ ((c >> 5) & 1)) << 2) + (c & 3); };
  float* plane = reinterpret_cast<float*>(smem + L::S0) + warp * TR * W;   // the warp's rows of the first plane
  {
    const float* ws = fb.ws + (size_t)blockIdx.z * 8 * MM + (size_t)(fl.par * 4) * MM;
    const bool vec = M % 4 == 0 && (!fl.first || (uintptr_t)d.in % 16 == 0);
    const float* nowhere = fl.first ? d.in : fb.ws;
    auto load = [&](float* dst, const float* g) {   // g: the plane at this warp's first row and the region's first column
      if (vec) {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int q = 0; q < (W + 127) / 128; ++q) {
            const int c = 4 * lane + 128 * q, i = ix0 + c, j = row0 + r;
            const bool in = c < W && i >= 0 && i < M && j >= 0 && j < M;
            if (c < W) cp_async16(dst + plane_at(r, c), in ? g + (long long)r * M + c : nowhere, in);
          }
      } else {
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int q = 0; q < TC; ++q) {
            const int c = lane + 32 * q, i = ix0 + c, j = row0 + r;
            const bool in = i >= 0 && i < M && j >= 0 && j < M;
            cp_async4(dst + plane_at(r, c), in ? g + (long long)r * M + c : nowhere, in);
          }
      }
    };
    const long long at = (long long)row0 * M + ix0;
    if (fl.first) {
      load(plane, d.in + at);
    } else {
      load(plane, ws + at);
      load(plane + L::PLANE, ws + MM + at);
      load(plane + 2 * L::PLANE, ws + 2 * MM + at);
      load(plane + 3 * L::PLANE, ws + 3 * MM + at);
    }
  }
  // a lane's words of row r in a plane, as pairs
  auto plane_read = [&](const float* pl, int r, f2 (&v)[H]) {
    float w[TC];
    if constexpr (TC % 4 == 0) {
#pragma unroll
      for (int c = 0; c < TC; c += 4)
        *reinterpret_cast<float4*>(w + c) = *reinterpret_cast<const float4*>(pl + plane_at(r, lane * TC + c));
    } else {
#pragma unroll
      for (int c = 0; c < TC; ++c) w[c] = pl[plane_at(r, lane * TC + c)];
    }
#pragma unroll
    for (int c = 0; c < H; ++c) v[c] = f2pack(w[c], w[c + H]);
  };
  auto plane_write = [&](float* pl, int r, const f2 (&v)[H]) {
    float w[TC];
#pragma unroll
    for (int c = 0; c < H; ++c) {
      w[c] = f2lo(v[c]);
      w[c + H] = f2hi(v[c]);
    }
    if constexpr (TC % 4 == 0) {
#pragma unroll
      for (int c = 0; c < TC; c += 4)
        *reinterpret_cast<float4*>(pl + plane_at(r, lane * TC + c)) = *reinterpret_cast<const float4*>(w + c);
    } else {
#pragma unroll
      for (int c = 0; c < TC; ++c) pl[plane_at(r, lane * TC + c)] = w[c];
    }
  };
#pragma unroll
  for (int c = 0; c < H; ++c) {
    float e0, w0, g0, e1, w1, g1;
    column_coefs(d, col0 + c, e0, w0, g0);
    column_coefs(d, col0 + c + H, e1, w1, g1);
    s.ce[c] = f2pack(e0, e1);
    s.cw[c] = f2pack(w0, w1);
    s.cgi[c] = f2pack(g0, g1);
  }
#pragma unroll
  for (int r = 0; r < TR; ++r) row_coefs(d, row0 + r, s.cs[r], s.cn[r], s.gj[r]);

  // Far-field data, in chunks of T steps, each evaluated a chunk ahead.  Lane l evaluates the far
  // column's value of step l / TR on the warp's row l % TR; the far row's T x W values are
  // spread over the cluster's threads and sent to the last CTA, whose last warp holds that row.
  const bool far_col = ix0 + L::W == M, far_row = jy0 + R == M;   // uniform over the cluster
  const bool owns_far_row = far_row && rank == C - 1 && warp == kFineWarps - 1;
  const bool owns_far_col = far_col && lane == 31;
  const int nstep = fl.nstep, step0 = fl.step0;
  float* fcol = reinterpret_cast<float*>(smem + L::FC) + warp * 64;   // [2 chunks][T][TR]
  auto far_chunk = [&](int chunk) {
    if (!far_col && !far_row) return;
    const int t = chunk * T + lane / TR, j = row0 + lane % TR;
    // (float)(tau0 + (step + 1) dtau) in FP64, once per lane and chunk
    const float tau = (float)(d.tau0 + (step0 + t + 1) * d.dtau);
    if (far_col)
      fcol[(chunk & 1) * 32 + lane] =
          t < nstep && j >= 0 ? far_field(pf, (float)(M - 1) * fb.h, (float)j * fb.h, tau) : 0.f;
    if (far_row) {
      const int slot = chunk % 3, n = min(T, nstep - chunk * T) * L::W;
      unsigned char* ff = smem + L::FF + (size_t)slot * T * WP * 8;
      if (owns_far_row && lane == 0) mbar_arm(far_mb + slot, n * 4);
      const uint32_t a = cluster_addr(smem_addr(ff), C - 1), m = cluster_addr(smem_addr(far_mb + slot), C - 1);
      for (int e = rank * kFineThreads + (int)threadIdx.x; e - lane < n; e += C * kFineThreads) {
        const int u = e / L::W, c = e % L::W, i = ix0 + c;   // a warp's nodes share u: W is a multiple of 32
        const float tt = __shfl_sync(0xffffffffu, tau, u * TR);
        st_async_f32(a + 4 * (u * WP * 2 + (c / TC) * L::HP * 2 + 2 * (c % TC % H) + c % TC / H),
                     i >= 0 ? far_field(pf, (float)i * fb.h, (float)(M - 1) * fb.h, tt) : 0.f, m);
      }
    }
    __syncwarp();
  };
  // Inverse diagonals, by way of the private words: a loop of four pairs of nodes at a time (executed once
  // per launch, its unrolled code would be fetched at several clocks per instruction; one
  // pair at a time waits for each reciprocal: 32 slices of 1024 x 1024, 128 steps, 22.7 ms against
  // 22.4).
#pragma unroll 4
  for (int e = 0; e < TR * H; ++e) {
    const int r = e / H, i0 = col0 + e - r * H, i1 = i0 + H, j = row0 + r;
    const bool in = j >= 0 && j < M - 1;
    s.dp[e] = f2pack(in && i0 >= 0 && i0 < M - 1 ? inv_diag(d, i0, j) : 0.f,
                     in && i1 >= 0 && i1 < M - 1 ? inv_diag(d, i1, j) : 0.f);
  }
  cp_async_wait_all();
  __syncwarp();
#pragma unroll
  for (int r = 0; r < TR; ++r) {
    plane_read(plane, r, s.hi[r]);
    f2 lo[H], dp[H];
    if (!fl.first) {
      plane_read(plane + L::PLANE, r, lo);
      plane_read(plane + 2 * L::PLANE, r, s.d[r]);
      plane_read(plane + 3 * L::PLANE, r, dp);
    }
#pragma unroll
    for (int c = 0; c < H; ++c) {
      s.iv[r][c] = s.dp[r * H + c];
      s.b[r][c] = 0;
      if (fl.first) s.d[r][c] = 0;
      s.lo[r * H + c] = fl.first ? 0 : lo[c];
      s.dp[r * H + c] = fl.first ? 0 : dp[c];
    }
  }
  // mbarriers are initialised and the staged rows read before the first row is published
  cluster_barrier(cluster, C);

  // The far-edge nodes move to step t of this launch: far_load fetches the far column's values,
  // far_set sets row r.
  float fv[TR];
  int ff_at = 0;   // slot of step t in the far row's ring of 3 T steps
  auto far_load = [&](int t) {
#pragma unroll
    for (int r = 0; r < TR; ++r) fv[r] = fcol[(t & (2 * T - 1)) * TR + r];
    if (owns_far_row) {
      const int chunk = t / T;
      ff_at = t % (3 * T);
      if (t % T == 0 && !s.dead) s.dead = !mbar_wait(far_mb + chunk % 3, (chunk / 3) & 1);
    }
  };
  auto far_set = [&](int r, bool on) {
    s.hi[r][H - 1] = f2pack(f2lo(s.hi[r][H - 1]), owns_far_col && on ? fv[r] : f2hi(s.hi[r][H - 1]));
    if (r == TR - 1 && owns_far_row && on) {
      const f2* ff = reinterpret_cast<const f2*>(smem + L::FF) + ff_at * WP + lane * L::HP;
#pragma unroll
      for (int c = 0; c < H; ++c) s.hi[TR - 1][c] = ff[c];
    }
  };

  const bool whole = nstep > 1;
  if (whole || min(fl.s_end, step_sweeps(d, step0)) > fl.s_begin) {   // (a split step's launch may have no sweep)
    far_chunk(0);
    far_load(0);
#pragma unroll
    for (int r = 0; r < TR; ++r) far_set(r, true);
    s.template publish<true, true>(0);
    s.template publish<true, false>(0);
    uint32_t q = 0;
    auto nothing = [](int) {};
    const int xstart = d.xstart, first_late = d.sweepsxl == 2 && whole ? d.xlate - step0 : 1 << 30;
    int t = 0;
    while (t < nstep) {
      if (t % T == 0) {
        // The next chunk of far-field data.  Its far row reuses the ring slot of the chunk two
        // before this one, whose last reader has entered the chunk before this one: the split
        // cluster barrier, a whole chunk long, orders the stores after that.
        const int chunk = t / T;
        const bool next = (chunk + 1) * T < nstep, next2 = (chunk + 2) * T < nstep;
        if (far_row && C > 1 && chunk >= 2 && next) cluster_wait();
        if (next) far_chunk(chunk + 1);
        if (far_row && C > 1 && chunk >= 1 && next2) cluster_arrive();
      }
      const int end = min(nstep, (t / T + 1) * T);
      if (t >= first_late) {
        // The late steps, nearly all of a long launch: two sweeps each, one down and one up.
        __syncthreads();
        for (; t < end; ++t, q += 2) {
          const bool more = t + 1 < nstep;
          s.template sweep<true, 0, true, true>(q, true, nothing);
          if (more) far_load(t + 1);
          s.template sweep<false, 2, false, true>(q + 1, more, [&](int r) { far_set(r, more); });
        }
        continue;
      }
      const int m_item = step_sweeps(d, step0 + t);
      const int sa = whole ? 0 : fl.s_begin, sb = whole ? m_item : min(fl.s_end, m_item);
      const bool ends = sb == m_item, extrap = step0 + t + 1 >= xstart, more = t + 1 < nstep;
      // first sweep, middle sweeps, and the sweep that ends the step (a piece of a split step
      // may lack it, or consist of it alone)
      const int mid = sb - sa - (ends ? 2 : 1);
      s.template sweep<true, 0, true, false>(q, more || (mid >= 0 && (ends || mid > 0)), nothing);
      ++q;
      for (int k = 0; k < mid; ++k, ++q)
        s.template sweep<false, 0, true, false>(q, more || ends || k + 1 < mid, nothing);
      ++t;
      if (!ends) continue;
      if (more) far_load(t);
      auto far = [&](int r) { far_set(r, more); };
      if (mid < 0) {   // the piece's one sweep ends its step: nothing follows in this launch
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          if (extrap) s.template commit<true>(r);
          else s.template commit<false>(r);
        }
      } else {
        if (extrap) s.template sweep<false, 2, true, false>(q, more, far);
        else s.template sweep<false, 1, true, false>(q, more, far);
        ++q;
      }
    }
  }
  if (s.dead && lane == 0) atomicOr(fb.status, 2);
  cluster_barrier(cluster, C);   // no CTA leaves while a neighbour may still store into it

  // the part of the region this launch leaves exact, coalesced along the rows
  const int i_lo = tx == 0 ? 0 : ix0 + fb.H, j_lo = ty == 0 ? 0 : jy0 + fb.H;
  const int i_hi = tx == fb.ntx - 1 ? M : region_origin(tx + 1, fb.ntx, L::W, M) + fb.H;
  const int j_hi = ty == fb.nty - 1 ? M : region_origin(ty + 1, fb.nty, R, M) + fb.H;
#pragma unroll
  for (int r = 0; r < TR; ++r) {
    f2 lo[H], dp[H];
#pragma unroll
    for (int c = 0; c < H; ++c) {
      lo[c] = s.lo[r * H + c];
      dp[c] = s.dp[r * H + c];
      if (fl.last) s.hi[r][c] = f2add(s.hi[r][c], lo[c]);
    }
    plane_write(plane, r, s.hi[r]);
    if (!fl.last) {
      plane_write(plane + L::PLANE, r, lo);
      plane_write(plane + 2 * L::PLANE, r, s.d[r]);
      plane_write(plane + 3 * L::PLANE, r, dp);
    }
  }
  __syncwarp();
  float* wo = fb.ws + (size_t)blockIdx.z * 8 * MM + (size_t)((fl.par ^ 1) * 4) * MM;
  const bool vec = M % 4 == 0 && (!fl.last || (uintptr_t)d.out % 16 == 0);
  auto store = [&](const float* src, float* g) {
    if (vec) {
#pragma unroll
      for (int r = 0; r < TR; ++r)
#pragma unroll
        for (int q = 0; q < (W + 127) / 128; ++q) {
          const int c = 4 * lane + 128 * q, i = ix0 + c, j = row0 + r;
          if (c < W && i >= i_lo && i < i_hi && j >= j_lo && j < j_hi)
            *reinterpret_cast<float4*>(g + (long long)r * M + c) = *reinterpret_cast<const float4*>(src + plane_at(r, c));
        }
    } else {
#pragma unroll
      for (int r = 0; r < TR; ++r)
#pragma unroll
        for (int q = 0; q < TC; ++q) {
          const int c = lane + 32 * q, i = ix0 + c, j = row0 + r;
          if (i >= i_lo && i < i_hi && j >= j_lo && j < j_hi) g[(long long)r * M + c] = src[plane_at(r, c)];
        }
    }
  };
  const long long at = (long long)row0 * M + ix0;
  if (fl.last) {
    store(plane, d.out + at);
  } else {
    store(plane, wo + at);
    store(plane + L::PLANE, wo + MM + at);
    store(plane + 2 * L::PLANE, wo + 2 * MM + at);
    store(plane + 3 * L::PLANE, wo + 3 * MM + at);
  }
}

// Launch and occupancy of one instance; the definitions below are instantiated once each, in the
// fine_w*.cu files.  spread: claim over half of an SM's shared memory, so that the CTAs of a
// launch that does not fill the GPU get an SM each.
template <int TC, int TR>
int fine_tile_launch(const FineBatch& fb, const FineLaunch& fl, bool spread, cudaStream_t s);
template <int TC, int TR>
int fine_tile_capacity(int C);   // clusters of C CTAs the device runs at once (0: unknown)

}  // namespace bsp
