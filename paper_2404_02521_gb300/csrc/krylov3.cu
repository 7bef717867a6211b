// Numerical coarse model G for three assets (Sec. 3.2 with n = 3): implicit-Euler steps whose
// systems are too stiff for Jacobi, solved by BiCGSTAB (van der Vorst 1992) on the
// Jacobi-scaled increment system D^{-1}(I - dtau R_h) d = D^{-1} dtau R_h u in FP32, one state.
// Each step starts from the previous step's increment; a breakdown restarts from the current
// iterate; a vanishing right-hand side gives d = 0.
//
// The whole propagation is one cooperative launch.  An iteration is two passes over the grid, each
// followed by one grid barrier that also carries its dot products:
//   A  r = s - omega t, p = r + beta (p - omega v), x += alpha p_old + omega s, v = A^ p:
//      (r^, v), (r, r)
//   B  s = r - alpha v, t = A^ s: (t, s), (t, t), (r^, s), (r^, t)
// The stencil's operand is formed while a tile is staged in shared memory, on the tile's halo
// too (from the vectors its owner wrote before the last barrier), so no barrier separates a vector
// update from the product that reads it; p and v alternate between two buffers because a
// neighbour may still read the old ones.  Every block adds the block sums in the same order
// and so takes the same decisions.
//
// What bounds it: the latency of two barriers and two rounds of L2 loads per iteration (the
// vectors of a 64^3 state are 1 MB each and stay in L2).  It replaces a chain of seven kernels per
// iteration with one-thread reductions and a host check every fourth: a slice of four steps at
// 64^3 takes 1.02 ms, 12.06 before.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "fine3.cuh"
#include "grid_barrier.cuh"

namespace bsp {

constexpr int kK3Attempts = 3;
constexpr int kK3Planes = 4;             // planes of k per tile: 256 tiles at 64^3
constexpr int kK3Threads = kF3TileI * kF3TileJ;
constexpr int kK3HI = kF3TileI + 2, kK3HJ = kF3TileJ + 2, kK3HK = kK3Planes + 2;
constexpr int kK3Tile = kK3HI * kK3HJ * kK3HK;
constexpr int kK3Ring = kK3HI * kK3HJ - kK3Threads;                       // halo entries of an inner plane
constexpr int kK3Halo = 2 * kK3HI * kK3HJ + kK3Planes * kK3Ring;          // halo entries of a tile

struct K3Words {
  float4 partials[2][kGridMaxBlocks];
  unsigned arrivals;   // zero at launch
};

struct K3Args {
  F3Batch fb;          // item 0: in, out, hi, lo, tau0
  float *x, *r, *rh, *s, *t;
  float *p[2], *v[2];
  K3Words* words;
  int* status;         // bit 0: no convergence, bit 1: a barrier timed out; the launch returns at once if set
  int nsteps, maxit;
  float tol;
};

__global__ void __launch_bounds__(kK3Threads, 2) k3_solve_kernel(const __grid_constant__ K3Args a) {
  __shared__ float sd[kK3Tile], sh[kK3Tile];
  if (*(volatile int*)a.status) return;   // an earlier launch of the solve failed (uniform)
  const F3Batch& fb = a.fb;
  const F3Item& it = fb.it[0];
  const int M = fb.M, sz = M * M;
  const int tiles_i = (M + kF3TileI - 1) / kF3TileI, tiles_j = (M + kF3TileJ - 1) / kF3TileJ;
  const int tiles = tiles_i * tiles_j * ((M + kK3Planes - 1) / kK3Planes);
  const int tid = threadIdx.y * kF3TileI + threadIdx.x;
  const int L0 = (kK3HJ + threadIdx.y + 1) * kK3HI + threadIdx.x + 1;   // tile index of the column's first plane
  constexpr int LZ = kK3HI * kK3HJ;
  const F3Coef& c = fb.c;
  GridGroup<kK3Threads> grid{&a.words->arrivals, a.words->partials[0], kGridMaxBlocks, a.status, (int)blockIdx.x, (int)gridDim.x, tid};

  int i0 = 0, j0 = 0, k0 = 0;
  // body() for each of this block's tiles, whose first node is (i0, j0, k0)
  auto each_tile = [&](auto&& body) {
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      const int tk = tile / (tiles_i * tiles_j), rem = tile - tk * (tiles_i * tiles_j), tj = rem / tiles_i;
      i0 = (rem - tj * tiles_i) * kF3TileI;
      j0 = tj * kF3TileJ;
      k0 = tk * kK3Planes;
      body();
    }
  };
  // node kk of the thread's column: f(kk, e, pde) where it lies in the grid
  auto column = [&](auto&& f) {
    const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
#pragma unroll
    for (int kk = 0; kk < kK3Planes; ++kk) {
      const int k = k0 + kk;
      if (i < M && j < M && k < M) f(kk, k * sz + j * M + i, i < M - 1 && j < M - 1 && k < M - 1);
    }
  };
  // f(q, e, in) for every halo entry q of the tile, e its node (0 where it lies outside the grid)
  auto halo = [&](auto&& f) {
#pragma unroll 2
    for (int h = tid; h < kK3Halo; h += kK3Threads) {
      int bi, bj, bk;
      if (h < 2 * LZ) {
        bk = h < LZ ? 0 : kK3HK - 1;
        const int w = h < LZ ? h : h - LZ;
        bj = w / kK3HI;
        bi = w - bj * kK3HI;
      } else {
        const int r = h - 2 * LZ, pl = r / kK3Ring, w = r - pl * kK3Ring;
        bk = pl + 1;
        if (w < 2 * kK3HI) {
          bj = w < kK3HI ? 0 : kK3HJ - 1;
          bi = w < kK3HI ? w : w - kK3HI;
        } else {
          bj = 1 + ((w - 2 * kK3HI) >> 1);
          bi = ((w - 2 * kK3HI) & 1) * (kK3HI - 1);
        }
      }
      const int i = i0 + bi - 1, j = j0 + bj - 1, k = k0 + bk - 1;
      const bool in = i >= 0 && i < M && j >= 0 && j < M && k >= 0 && k < M;
      f((bk * kK3HJ + bj) * kK3HI + bi, in ? k * sz + j * M + i : 0, in);
    }
  };
  // the tile's entries of the thread's column that lie outside the grid are zero
  auto clear = [&](float* t) {
    const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
#pragma unroll
    for (int kk = 0; kk < kK3Planes; ++kk)
      if (i >= M || j >= M || k0 + kk >= M) t[L0 + kk * LZ] = 0.f;
  };
  struct Stencil {
    F3Col w;
    float dxy;
  };
  auto stencil = [&]() {
    const float fi = (float)(i0 + (int)threadIdx.x), fj = (float)(j0 + (int)threadIdx.y);
    const float ax = c.A[0] * (fi * fi), ay = c.A[1] * (fj * fj), mx = c.D[0] * fi, my = c.D[1] * fj;
    return Stencil{{ax + mx, ax - mx, ay + my, ay - my, c.Cxy * (fi * fj), c.Cxz * fi, c.Cyz * fj},
                   1.0f + 2.0f * (ax + ay) + c.rdt};
  };
  // off-diagonal sum and diagonal at plane kk of the column
  auto apply = [&](const float* t, const Stencil& st, int kk, float& diag) {
    const float fk = (float)(k0 + kk), az = c.A[2] * (fk * fk), mz = c.D[2] * fk;
    diag = st.dxy + 2.0f * az;
    return f3_tile_offdiag<kK3HI, kK3HJ>(t, L0 + kk * LZ, st.w, az, mz, fk);
  };

  for (int step = 0; step < a.nsteps; ++step) {
    // the state with the previous step's increment, and the far faces of this step
    const float tau_new = it.tau0 + (step + 1) * fb.dtau;
    each_tile([&] {
      column([&](int kk, int e, bool pde) {
        float hi, lo = 0.f;
        if (step == 0) {
          hi = it.in[e];
          a.x[e] = 0.f;
        } else {
          hi = it.hi[e];
          lo = it.lo[e];
          const float v = a.x[e];
          const float sm = hi + v, bb = sm - hi;
          const float l = lo + ((hi - (sm - bb)) + (v - bb));
          hi = sm + l;
          lo = l - (hi - sm);
        }
        if (!pde) hi = f3_far_field(fb, i0 + threadIdx.x, j0 + threadIdx.y, k0 + kk, tau_new);
        it.hi[e] = hi;
        it.lo[e] = lo;
      });
    });
    grid.barrier();
    bool conv = false, fail = true;
    for (int attempt = 0; attempt < kK3Attempts && !conv && fail && !grid.dead; ++attempt) {
      // b^ = D^{-1} dtau R_h u, r = r^ = p = b^ - A^ x
      float sums[4] = {0.f, 0.f, 0.f, 0.f};
      each_tile([&] {
        clear(sd);
        clear(sh);
        column([&](int kk, int e, bool) {
          sd[L0 + kk * LZ] = __ldcg(a.x + e);
          sh[L0 + kk * LZ] = __ldcg(it.hi + e);
        });
        halo([&](int q, int e, bool in) {
          sd[q] = in ? __ldcg(a.x + e) : 0.f;
          sh[q] = in ? __ldcg(it.hi + e) : 0.f;
        });
        __syncthreads();
        const Stencil st = stencil();
        column([&](int kk, int e, bool pde) {
          float r = 0.f, bh = 0.f;
          if (pde) {
            float diag;
            const float o = apply(sh, st, kk, diag);
            const float b = o - (diag - 1.0f) * sh[L0 + kk * LZ], invd = 1.0f / diag;
            bh = invd * b;
            r = bh - (sd[L0 + kk * LZ] - invd * apply(sd, st, kk, diag));
          }
          a.r[e] = r;
          a.rh[e] = r;
          a.p[0][e] = r;
          sums[0] = fmaf(bh, bh, sums[0]);
          sums[1] = fmaf(r, r, sums[1]);
        });
        __syncthreads();
      });
      grid.sum(sums);
      float rho = sums[1];
      const float stop2 = a.tol * a.tol * sums[0];
      const bool zero = !(sums[0] > 1e-30f);
      conv = sums[1] <= stop2 || zero;
      fail = false;
      if (zero) each_tile([&] { column([&](int, int e, bool) { a.x[e] = 0.f; }); });
      float alpha = 0.f, omega = 0.f, beta = 0.f;
      bool pending = false;
      for (int itn = 0; !conv && !grid.dead;) {
        // pass A; the first one of an attempt has its r and p (buffer 0) already
        const float* vo = a.v[itn ? (itn - 1) & 1 : 0];
        const float* po = a.p[itn ? (itn - 1) & 1 : 0];
        float* vn = a.v[itn & 1];
        float* pn = a.p[itn & 1];
        float sa[4] = {0.f, 0.f, 0.f, 0.f};
        auto next_p = [&](int e, float& r) {
          r = fmaf(-omega, __ldcg(a.t + e), __ldcg(a.s + e));
          return fmaf(beta, fmaf(-omega, __ldcg(vo + e), __ldcg(po + e)), r);
        };
        each_tile([&] {
          clear(sd);
          column([&](int kk, int e, bool) {
            float p, r;
            if (itn) {
              p = next_p(e, r);
              a.x[e] += alpha * po[e] + omega * a.s[e];
              a.r[e] = r;
              pn[e] = p;
              sa[1] = fmaf(r, r, sa[1]);
            } else {
              p = __ldcg(po + e);
            }
            sd[L0 + kk * LZ] = p;
          });
          halo([&](int q, int e, bool in) {
            float r;
            sd[q] = in ? (itn ? next_p(e, r) : __ldcg(po + e)) : 0.f;
          });
          __syncthreads();
          const Stencil st = stencil();
          column([&](int kk, int e, bool pde) {
            float v = 0.f;
            if (pde) {
              float diag;
              const float o = apply(sd, st, kk, diag);
              v = sd[L0 + kk * LZ] - o * (1.0f / diag);
            }
            vn[e] = v;
            sa[0] = fmaf(a.rh[e], v, sa[0]);
          });
          __syncthreads();
        });
        grid.sum(sa);
        if (itn) {
          conv = sa[1] <= stop2;
          if (conv) break;
          if (pending) fail = true;
          if (fail || itn == a.maxit) break;
        }
        if (sa[0] == 0.f) {
          fail = true;
          break;
        }
        alpha = rho / sa[0];
        // pass B
        float sb[4] = {0.f, 0.f, 0.f, 0.f};
        each_tile([&] {
          clear(sd);
          column([&](int kk, int e, bool) {
            const float s = fmaf(-alpha, vn[e], a.r[e]);
            a.s[e] = s;
            sd[L0 + kk * LZ] = s;
          });
          halo([&](int q, int e, bool in) { sd[q] = in ? fmaf(-alpha, __ldcg(vn + e), __ldcg(a.r + e)) : 0.f; });
          __syncthreads();
          const Stencil st = stencil();
          column([&](int kk, int e, bool pde) {
            const float s = sd[L0 + kk * LZ], rh = a.rh[e];
            float t = 0.f;
            if (pde) {
              float diag;
              const float o = apply(sd, st, kk, diag);
              t = s - o * (1.0f / diag);
            }
            a.t[e] = t;
            sb[0] = fmaf(t, s, sb[0]);
            sb[1] = fmaf(t, t, sb[1]);
            sb[2] = fmaf(rh, s, sb[2]);
            sb[3] = fmaf(rh, t, sb[3]);
          });
          __syncthreads();
        });
        grid.sum(sb);
        omega = sb[1] > 0.f ? sb[0] / sb[1] : 0.f;
        const float rho_new = sb[2] - omega * sb[3];
        if (omega == 0.f || rho == 0.f) {
          pending = true;   // finish this iteration, then restart
          beta = 0.f;
        } else {
          beta = (rho_new / rho) * (alpha / omega);
          rho = rho_new;
        }
        ++itn;
      }
    }
    if (!conv || grid.dead) {
      if (blockIdx.x == 0 && tid == 0 && !grid.dead) atomicOr(a.status, 1);
      return;
    }
  }
  each_tile([&] {
    column([&](int, int e, bool) {
      const float h0 = it.hi[e], v = a.x[e], sm = h0 + v, bb = sm - h0;
      const float l = it.lo[e] + ((h0 - (sm - bb)) + (v - bb));
      const float hn = sm + l;
      it.out[e] = hn + (l - (hn - sm));
    });
  });
}

// Blocks of the solver that the current device runs at once, measured once per device.
static int k3_blocks(int* out) {
  static std::mutex mu;
  static int known[64] = {};
  int dev = 0;
  BS_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (dev >= 64 || !known[dev]) {
    int per_sm = 0, sms = 0;
    BS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k3_solve_kernel, kK3Threads, 0));
    BS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int n = std::min(per_sm * sms, kGridMaxBlocks);
    if (n < 1) return set_error(BS_ERR_CUDA, "three-asset coarse solver: no block fits an SM");
    if (dev >= 64) {
      *out = n;
      return BS_OK;
    }
    known[dev] = n;
  }
  *out = known[dev];
  return BS_OK;
}

constexpr int kK3Vectors = 11;
size_t k3_workspace_bytes(int M) {
  const size_t n3 = (size_t)M * M * M;
  return ((kK3Vectors * n3 * sizeof(float) + 255) & ~(size_t)255) + sizeof(K3Words) + 256;
}
int* k3_status(void* ws, int M) {
  return reinterpret_cast<int*>(static_cast<unsigned char*>(ws) + k3_workspace_bytes(M) - 256);
}

// G over one slice for one state: nsteps implicit steps of size dtau from tau0, each solved by
// BiCGSTAB to relative residual tol (at most maxit iterations per attempt).  Asynchronous; the
// outcome is or-ed into k3_status(ws), zero before the first call, and a call that finds it set
// does nothing.
int coarse_propagate3_krylov(int M, double xmax, const bs_params3& p, const float* u_in, float* u_out, double tau0,
                             double dtau, int nsteps, double tol, int maxit, void* ws, cudaStream_t s) {
  const size_t n3 = (size_t)M * M * M;
  int blocks = 0;
  int rc = k3_blocks(&blocks);
  if (rc) return rc;
  float* f = static_cast<float*>(ws);
  K3Args a;
  a.fb = f3_batch(M, xmax, p, dtau);
  a.fb.n = 1;
  F3Item& it = a.fb.it[0];
  it.in = u_in;
  it.out = u_out;
  it.tau0 = (float)tau0;
  float** v[kK3Vectors] = {&it.hi, &it.lo, &a.x, &a.r, &a.rh, &a.s, &a.t, &a.p[0], &a.p[1], &a.v[0], &a.v[1]};
  for (int q = 0; q < kK3Vectors; ++q) *v[q] = f + q * n3;
  a.status = k3_status(ws, M);
  a.words = reinterpret_cast<K3Words*>(reinterpret_cast<unsigned char*>(a.status) - sizeof(K3Words));
  a.nsteps = nsteps;
  a.maxit = maxit;
  a.tol = (float)tol;
  const int tiles = ((M + kF3TileI - 1) / kF3TileI) * ((M + kF3TileJ - 1) / kF3TileJ) * ((M + kK3Planes - 1) / kK3Planes);
  BS_CUDA_TRY(cudaMemsetAsync(&a.words->arrivals, 0, sizeof(unsigned), s));
  void* args[] = {&a};
  BS_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k3_solve_kernel), dim3(std::min(tiles, blocks)),
                                          dim3(kF3TileI, kF3TileJ), args, 0, s));
  return BS_OK;
}

// The outcome of the calls since the status was zeroed (synchronous).
int k3_result(void* ws, int M, int maxit, cudaStream_t s) {
  int h = 0;
  BS_CUDA_TRY(cudaMemcpyAsync(&h, k3_status(ws, M), sizeof(int), cudaMemcpyDeviceToHost, s));
  BS_CUDA_TRY(cudaStreamSynchronize(s));
  if (h & 2) return set_error(BS_ERR_CUDA, "three-asset coarse BiCGSTAB: a grid barrier timed out");
  if (h) return set_error(BS_ERR_NOCONV, "three-asset coarse BiCGSTAB: no convergence within %d iterations", maxit);
  return BS_OK;
}

}  // namespace bsp

using namespace bsp;

extern "C" int coarse_propagate3(int M, double xmax, const bs_params3* p, const float* u_in, float* u_out,
                                 double tau0, double dtau_slice, int nsteps, bs_stream stream) {
  int rc = f3_check(M, xmax, p);
  if (rc) return rc;
  if (!u_in || !u_out) return set_error(BS_ERR_ARG, "coarse_propagate3: NULL state");
  if (!(dtau_slice > 0.0) || nsteps < 1)
    return set_error(BS_ERR_ARG, "coarse_propagate3: dtau_slice=%g nsteps=%d", dtau_slice, nsteps);
  cudaStream_t s = (cudaStream_t)stream;
  void* ws = nullptr;
  note_device_alloc();
  BS_CUDA_TRY(cudaMallocAsync(&ws, k3_workspace_bytes(M), s));
  cudaError_t e = cudaMemsetAsync(k3_status(ws, M), 0, sizeof(int), s);
  rc = e == cudaSuccess ? BS_OK : cuda_error(e, "coarse_propagate3");
  if (!rc)
    rc = coarse_propagate3_krylov(M, xmax, *p, u_in, u_out, tau0, dtau_slice / nsteps, nsteps, g_opt.krylov_tol,
                                  g_opt.krylov_maxit, ws, s);
  if (!rc) rc = k3_result(ws, M, g_opt.krylov_maxit, s);
  cudaFreeAsync(ws, s);
  return rc;
}
