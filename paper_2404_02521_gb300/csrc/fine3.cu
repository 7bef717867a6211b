// F for three assets: eq. (bse_general) with n = 3, discretised like eq. (fd) (second
// differences along each axis, four-point cross differences for each pair, centred first
// differences: a 19-point stencil) and stepped by implicit Euler, for B states at once.
//
// Each step solves (I - dtau R_h) d = dtau R_h u (increment form, far-face Dirichlet data at
// the new time level) by Jacobi sweeps whose count follows from the Gershgorin bound q of the
// system (q < 0.8) and from how the step's solve starts (f3_sweeps): the first step from d = 0, the
// second from the previous increment, later ones from the extrapolation of the previous two.  u is
// carried as a compensated (hi, lo) FP32 pair.  Starting every step from the previous
// increment took 22 sweeps per step at q = 0.72 (64^3, dtau = 1/640) where the extrapolation
// takes 19 falling to 5: 16 states, 40 steps, 24.0 -> 11.0 ms, with the same error against 64
// bits (1.6e-6; 3.6e-6 and 2.2e-6 on longer runs, all unchanged to three digits).
// Stencil coefficients are products of host-rounded FP32 constants and exact integer node
// indices (x_p = i_p h, so h cancels).
//
// One launch of f3_sweep_kernel per Jacobi sweep.  A block owns kF3TileI x kF3TileJ columns
// (i, j) and kF3PlanesPerBlock planes k; it stages the halo tile of the old increment (one
// node on every side, zero outside the grid) in shared memory with asynchronous 4-byte copies
// that are all in flight at once, and loads its columns' own operands (b, and for the last
// sweep hi and lo) into registers before its single barrier.  Each thread then walks its
// column (i, j) up through the block's planes.  The first sweep of a step also stages hi and
// forms b = dtau R_h hi (the RHS phase); the last sweep also adds the increment to (hi, lo)
// (APPLY) and writes the far faces of the next step (FACE).  So a step is its sweeps alone;
// f3_phase_kernel remains only for the passes before the first step (INIT) and after the last (OUT).
//
// Layout: u[(k*M + j)*M + i] with i the index of asset 1 (fastest), j of asset 2, k of
// asset 3.  Nodes with an index M - 1 carry Dirichlet data; nodes with an index 0 carry the
// PDE row itself (every coefficient that would reach index -1 is a multiple of that index).
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "fine3.cuh"

namespace bsp {

// The pointwise passes of a propagation: INIT copies u_in into (hi, lo = 0), zeroes the increment
// and its history and sets the far faces of the first step; OUT writes hi + lo.
enum { F3_INIT = 0, F3_OUT = 1 };
__global__ void __launch_bounds__(kF3Threads) f3_phase_kernel(const __grid_constant__ F3Batch fb, int phase, int nsteps) {
  const F3Item& it = fb.it[blockIdx.y];
  const int M = fb.M, n3 = M * M * M;
  const int e = blockIdx.x * kF3Threads + threadIdx.x;
  if (e >= n3) return;
  if (phase == F3_OUT) {
    it.out[e] = it.hi[e] + it.lo[e];
    return;
  }
  int i, j, k;
  f3_node(e, M, i, j, k);
  const bool pde = i < M - 1 && j < M - 1 && k < M - 1;
  it.hi[e] = pde || nsteps == 0 ? it.in[e] : f3_far_field(fb, i, j, k, it.tau0 + fb.dtau);
  it.lo[e] = 0.f;
  it.dA[e] = 0.f;
  it.dB[e] = 0.f;
  it.dP[e] = 0.f;
}

// Asynchronous 4-byte global -> shared copy (all of a thread's copies in flight at once);
// with ok == false the destination is zero-filled and nothing is read.
__device__ __forceinline__ void f3_cp_async4(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
}

// Halo tile of one block: kF3TileI x kF3TileJ columns and kF3PlanesPerBlock planes plus one
// node on every side, i fastest.  Entries outside the grid are 0 (their weights are 0 too).
constexpr int kHI = kF3TileI + 2, kHJ = kF3TileJ + 2, kHK = kF3PlanesPerBlock + 2;
constexpr int kTileFloats = kHI * kHJ * kHK;

// One Jacobi sweep: d_new = (b + offdiag(d_old)) / diag at PDE nodes, 0 elsewhere.  A block
// stages its halo tile of d_old in shared memory (asynchronous copies, coalesced along i),
// then each thread walks its column (i, j) up through the block's planes.  The first sweep of
// a step also stages the state and forms b = dtau R_h hi (RHS); the last one also adds its
// increment to (hi, lo) (APPLY) and writes the far faces of step face_step (FACE; -1: none).
// A step has at least two sweeps, so no launch both reads the state's neighbours and writes
// the state.
enum { F3S_FIRST = 1, F3S_LAST = 2 };
template <int FLAGS>
__global__ void __launch_bounds__(kF3TileI * kF3TileJ, 4) f3_sweep_kernel(const __grid_constant__ F3Batch fb,
                                                                         int cur, int tiles_i, int face_step,
                                                                         int extrap) {
  constexpr bool first = FLAGS & F3S_FIRST, last = FLAGS & F3S_LAST;
  __shared__ float sd[kTileFloats];
  __shared__ float sh[first ? kTileFloats : 1];
  const F3Item& it = fb.it[blockIdx.z];
  const int M = fb.M;
  const int tj = blockIdx.x / tiles_i;   // uniform per block
  const int i0 = (blockIdx.x - tj * tiles_i) * kF3TileI, j0 = tj * kF3TileJ;
  const int k0 = blockIdx.y * kF3PlanesPerBlock;
  const float* __restrict__ din = cur ? it.dB : it.dA;
  float* __restrict__ dout = cur ? it.dA : it.dB;
  const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
  const int col = j * M + i, sz = M * M;
  const bool active = i < M && j < M, pdecol = i < M - 1 && j < M - 1;
  // the column's own operands for every plane, loaded with the tile (no load waits per plane)
  float bq[kF3PlanesPerBlock], hq[last ? kF3PlanesPerBlock : 1], lq[last ? kF3PlanesPerBlock : 1],
      pq[last ? kF3PlanesPerBlock : 1];
#pragma unroll
  for (int kk = 0; kk < kF3PlanesPerBlock; ++kk) {
    const int k = k0 + kk, e = k * sz + col;
    const bool pde = pdecol && k < M - 1;
    if (!first) bq[kk] = pde ? __ldg(it.b + e) : 0.f;
    if (last) {
      hq[kk] = pde ? it.hi[e] : 0.f;
      lq[kk] = pde ? it.lo[e] : 0.f;
      pq[kk] = pde ? it.dP[e] : 0.f;
    }
  }
  for (int q = threadIdx.y * kF3TileI + threadIdx.x; q < kTileFloats; q += kF3TileI * kF3TileJ) {
    const int ck = q / (kHI * kHJ);
    const int rem = q - ck * (kHI * kHJ);
    const int bj = rem / kHI;
    const int gi = i0 - 1 + (rem - bj * kHI), gj = j0 - 1 + bj, gk = k0 - 1 + ck;
    const bool in = gi >= 0 && gi < M && gj >= 0 && gj < M && gk >= 0 && gk < M;
    const int ge = in ? (gk * M + gj) * M + gi : 0;
    f3_cp_async4(sd + q, din + ge, in);
    if (first) f3_cp_async4(sh + q, it.hi + ge, in);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();   // the only barrier: threads outside the grid leave after it
  if (!active) return;
  const int k1 = min(k0 + kF3PlanesPerBlock, M);
  const bool face = last && face_step >= 0;
  const float tau_face = it.tau0 + (face_step + 1) * fb.dtau;
  if (!pdecol) {   // far-face column: no unknowns
    for (int k = k0; k < k1; ++k) {
      dout[k * sz + col] = 0.f;
      if (face) it.hi[k * sz + col] = f3_far_field(fb, i, j, k, tau_face);
    }
    return;
  }
  const F3Coef& c = fb.c;
  const float fi = (float)i, fj = (float)j;
  const float ax = c.A[0] * (fi * fi), ay = c.A[1] * (fj * fj);
  const float mx = c.D[0] * fi, my = c.D[1] * fj;
  const F3Col w = {ax + mx, ax - mx, ay + my, ay - my, c.Cxy * (fi * fj), c.Cxz * fi, c.Cyz * fj};
  const float dxy = 1.0f + 2.0f * (ax + ay) + c.rdt;
  const int L0 = (1 * kHJ + threadIdx.y + 1) * kHI + threadIdx.x + 1;   // tile index of plane k0
#pragma unroll
  for (int kk = 0; kk < kF3PlanesPerBlock; ++kk) {
    const int k = k0 + kk;
    if (k >= k1) break;
    const int e = k * sz + col;
    if (k == M - 1) {
      dout[e] = 0.f;   // far face
      if (face) it.hi[e] = f3_far_field(fb, i, j, k, tau_face);
      break;
    }
    const int L = L0 + kk * (kHI * kHJ);
    const float fk = (float)k;
    const float az = c.A[2] * (fk * fk), mz = c.D[2] * fk;
    const float diag = dxy + 2.0f * az;
    float bv;
    if (first) {   // RHS: b = offdiag(hi) - (diag - 1) hi
      bv = f3_tile_offdiag<kHI, kHJ>(sh, L, w, az, mz, fk) - (diag - 1.0f) * sh[L];
      it.b[e] = bv;
    } else {
      bv = bq[kk];
    }
    const float dn = (bv + f3_tile_offdiag<kHI, kHJ>(sd, L, w, az, mz, fk)) / diag;
    dout[e] = last && extrap ? fmaf(2.f, dn, -pq[kk]) : dn;
    if (last) {   // APPLY: compensated add of the increment, which the next step's guess extrapolates
      it.dP[e] = dn;
      const float h0 = hq[kk];
      const float sm = h0 + dn, bb = sm - h0;
      const float err = (h0 - (sm - bb)) + (dn - bb);
      const float l = lq[kk] + err;
      const float hn = sm + l;
      it.lo[e] = l - (hn - sm);
      it.hi[e] = hn;
    }
  }
}

// Gershgorin bound of I - dtau R_h over the PDE nodes: max of sum |off-diagonal| / diagonal.
static double f3_contraction_scan(int M, const bs_params3& p, double dtau) {
  double q = 0.0;
  const double rho[3][3] = {{1.0, p.rho[0], p.rho[1]}, {p.rho[0], 1.0, p.rho[2]}, {p.rho[1], p.rho[2], 1.0}};
  for (int k = 0; k <= M - 2; ++k)
    for (int j = 0; j <= M - 2; ++j)
      for (int i = 0; i <= M - 2; ++i) {
        const int id[3] = {i, j, k};
        double off = 0.0, diag = 1.0 + dtau * p.r;
        for (int a = 0; a < 3; ++a) {
          const double dif = 0.5 * p.sigma[a] * p.sigma[a] * id[a] * id[a], drift = 0.5 * p.r * id[a];
          off += std::fabs(dif + drift) + std::fabs(dif - drift);
          diag += dtau * 2.0 * dif;
        }
        for (int a = 0; a < 3; ++a)
          for (int b = a + 1; b < 3; ++b)
            off += 4.0 * std::fabs(0.25 * rho[a][b] * p.sigma[a] * p.sigma[b]) * id[a] * id[b];
        q = std::fmax(q, dtau * off / diag);
      }
  return q;
}

// jacobi_skew (capi.cu) for three assets.
static double f3_skew(int M, const bs_params3& p, double dtau) {
  const int pair[3][2] = {{0, 1}, {0, 2}, {1, 2}};
  double cross[3] = {0.0, 0.0, 0.0}, bound = 0.0;
  for (int c = 0; c < 3; ++c) {
    const double g = 0.25 * std::fabs(p.rho[c]) * p.sigma[pair[c][0]] * p.sigma[pair[c][1]] * dtau;
    cross[pair[c][0]] += g;
    cross[pair[c][1]] += g;
    bound += g;
  }
  for (int x = 0; x < 3; ++x) {
    const double a = 0.5 * p.sigma[x] * p.sigma[x] * dtau, c = std::fabs(0.5 * p.r * dtau - a) + cross[x];
    double s = c;
    for (int i = 1; i <= M - 2; ++i) s = std::fmax(s, 2.0 * i * c / (1.0 + 2.0 * a * (i - 1.0) * (i - 1.0)));
    bound += s;
  }
  return bound;
}

// The scan visits (M-1)^3 nodes (milliseconds at 128^3), and parareal_solve3 asks for the same
// bound on every F call: the last few results are kept per (M, parameters, dtau).
double f3_contraction(int M, const bs_params3& p, double dtau) {
  struct Entry {
    double key[9];
    double q;
  };
  static std::mutex mu;
  static Entry cache[8];
  static int used = 0, next = 0;
  const double key[9] = {(double)M, p.sigma[0], p.sigma[1], p.sigma[2], p.rho[0], p.rho[1], p.rho[2], p.r, dtau};
  {
    std::lock_guard<std::mutex> lock(mu);
    for (int e = 0; e < used; ++e)
      if (std::memcmp(cache[e].key, key, sizeof(key)) == 0) return cache[e].q;
  }
  const double q = f3_contraction_scan(M, p, dtau);
  std::lock_guard<std::mutex> lock(mu);
  std::memcpy(cache[next].key, key, sizeof(key));
  cache[next].q = q;
  next = (next + 1) % 8;
  used = used < 8 ? used + 1 : 8;
  return q;
}

// Sweeps of step `step` of a propagation, by how its solve starts: from zero, from the
// previous increment, or from the extrapolation of the previous two.  An extrapolated start is
// off by a mode's second difference in time, and the modes that have survived n steps decay by
// about 1/n per step, so the reduction that the solve owes falls with n, at first with n^2.  On
// white-noise states of 17^3 to 64^3, 4 to 80 steps at q = 0.72, the error is within 3.5% of the
// one with every step from the previous increment to 2^-10 (1.26e-7 after 4 steps at 17^3, 9.8e-7
// after 40 at 24^3, 1.80e-6 at 48^3; on payoffs the same to three digits).  n / 128 without the
// quadratic start takes a tenth fewer sweeps and left 2.8e-7 after those 4 steps; a fixed 2^-6 up to
// step 16 and 1/2 from there a fifth fewer, and 6e-6 after 40 at 24^3.  A target above 1/4
// takes an even count: the error recurrence e_{t+1} = l^m (2 e_t - e_{t-1}) of an extrapolated
// start has a root beyond 1 where l^m < -1/3 (l an eigenvalue of the sweep, which can be
// negative).
// Complex eigenvalues (drift above diffusion; skew bounds their imaginary part) need more, see
// extrap_stable.
constexpr int kF3ExtrapStart = 2;
static int f3_sweeps(double q, double skew, int step) {
  const double target = step == 0               ? 1.0 / 4194304.0
                        : step < kF3ExtrapStart ? 1.0 / 1024.0
                                                : std::fmin(std::fmin(step * step / 2048.0, step / 192.0), 0.5);
  if (q <= 0.0) return 2;
  const int m = std::max(2, (int)std::ceil(std::log(target) / std::log(q)));
  return step < kF3ExtrapStart ? m : extrap_sweeps(q, skew, target > 0.25 ? (m + 1) & ~1 : m);
}

int f3_check(int M, double xmax, const bs_params3* p) {
  if (!p) return set_error(BS_ERR_ARG, "params3 is NULL");
  if (M < 4 || M > 128) return set_error(BS_ERR_ARG, "three-asset grid: M=%d out of [4, 128]", M);
  if (!(xmax > 0.0)) return set_error(BS_ERR_ARG, "three-asset grid: xmax must be > 0");
  for (int a = 0; a < 3; ++a) {
    if (!(p->sigma[a] > 0.0)) return set_error(BS_ERR_ARG, "sigma must be > 0");
    if (!(std::fabs(p->rho[a]) < 1.0)) return set_error(BS_ERR_ARG, "|rho| must be < 1");
  }
  // the correlation matrix must be positive definite (its determinant, the 2x2 minors are
  // positive already)
  const double r12 = p->rho[0], r13 = p->rho[1], r23 = p->rho[2];
  if (!(1.0 - r12 * r12 - r13 * r13 - r23 * r23 + 2.0 * r12 * r13 * r23 > 0.0))
    return set_error(BS_ERR_ARG, "the correlation matrix is not positive definite");
  if (!(p->r >= 0.0)) return set_error(BS_ERR_ARG, "r must be >= 0");
  if (p->payoff != BS_PAYOFF_BASKET && p->payoff != BS_PAYOFF_EXCHANGE)
    return set_error(BS_ERR_ARG, "three-asset payoff must be BS_PAYOFF_BASKET or BS_PAYOFF_EXCHANGE");
  if (p->reserved != 0) return set_error(BS_ERR_ARG, "bs_params3.reserved must be 0");
  return BS_OK;
}

F3Batch f3_batch(int M, double xmax, const bs_params3& p, double dtau) {
  F3Batch fb = {};
  fb.M = M;
  fb.h = (float)(xmax / (M - 1));
  for (int a = 0; a < 3; ++a) {
    fb.c.A[a] = (float)(0.5 * p.sigma[a] * p.sigma[a] * dtau);
    fb.c.D[a] = (float)(0.5 * p.r * dtau);
    fb.w[a] = (float)p.w[a];
  }
  fb.c.Cxy = (float)(0.25 * p.rho[0] * p.sigma[0] * p.sigma[1] * dtau);
  fb.c.Cxz = (float)(0.25 * p.rho[1] * p.sigma[0] * p.sigma[2] * dtau);
  fb.c.Cyz = (float)(0.25 * p.rho[2] * p.sigma[1] * p.sigma[2] * dtau);
  fb.c.rdt = (float)(p.r * dtau);
  fb.kind = p.payoff;
  fb.K = (float)p.strike;
  fb.r = (float)p.r;
  fb.dtau = (float)dtau;
  fb.ex = PayoffF{};
  fb.ex.kind = BS_PAYOFF_EXCHANGE;
  fb.ex.s1 = (float)p.sigma[0];
  fb.ex.s2 = (float)p.sigma[1];
  fb.ex.rho = (float)p.rho[0];
  fb.ex.r = (float)p.r;
  return fb;
}

__global__ void f3_payoff_kernel(float* u, int M, float h, int kind, float w0, float w1, float w2, float K) {
  const int n3 = M * M * M;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n3) return;
  int i, j, k;
  f3_node(e, M, i, j, k);
  const float x = i * h, y = j * h, z = k * h;
  u[e] = kind == BS_PAYOFF_BASKET ? fmaxf(w0 * x + w1 * y + w2 * z - K, 0.f) : fmaxf(x - y, 0.f);
}

}  // namespace bsp

using namespace bsp;

extern "C" {

int bs_payoff3(int M, double xmax, const bs_params3* p, float* u, bs_stream stream) {
  int rc = f3_check(M, xmax, p);
  if (rc) return rc;
  if (!u) return set_error(BS_ERR_ARG, "bs_payoff3: NULL state");
  const int n3 = M * M * M;
  f3_payoff_kernel<<<(n3 + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      u, M, (float)(xmax / (M - 1)), p->payoff, (float)p->w[0], (float)p->w[1], (float)p->w[2], (float)p->strike);
  BS_CUDA_TRY(cudaGetLastError());
  return BS_OK;
}

int fine_propagate3(int M, double xmax, const bs_params3* p, const float* const* u_in, float* const* u_out,
                    const double* tau0, int B, double dtau, int nsteps, bs_stream stream) {
  int rc = f3_check(M, xmax, p);
  if (rc) return rc;
  if (!u_in || !u_out || !tau0) return set_error(BS_ERR_ARG, "fine_propagate3: NULL argument");
  if (B < 1 || nsteps < 0) return set_error(BS_ERR_ARG, "fine_propagate3: B=%d nsteps=%d", B, nsteps);
  if (!(dtau > 0.0)) return set_error(BS_ERR_ARG, "fine_propagate3: dtau <= 0");
  for (int b = 0; b < B; ++b)
    if (!u_in[b] || !u_out[b]) return set_error(BS_ERR_ARG, "fine_propagate3: NULL state %d", b);
  const double q = f3_contraction(M, *p, dtau);
  if (!(q < 0.8))
    return set_error(BS_ERR_ARG, "fine_propagate3: Jacobi bound %.3f >= 0.8 (take smaller steps)", q);
  const double skew = f3_skew(M, *p, dtau);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t n3 = (size_t)M * M * M;
  const unsigned blocks = (unsigned)((n3 + kF3Threads - 1) / kF3Threads);
  for (int base = 0; base < B; base += kF3MaxItems) {
    const int nb = B - base < kF3MaxItems ? B - base : kF3MaxItems;
    float* ws = nullptr;
    note_device_alloc();
    BS_CUDA_TRY(cudaMallocAsync((void**)&ws, (size_t)nb * 6 * n3 * sizeof(float), s));
    F3Batch fb = f3_batch(M, xmax, *p, dtau);
    fb.n = nb;
    for (int t = 0; t < nb; ++t) {
      F3Item& it = fb.it[t];
      float* w = ws + (size_t)t * 6 * n3;
      it.in = u_in[base + t];
      it.out = u_out[base + t];
      it.hi = w;
      it.lo = w + n3;
      it.b = w + 2 * n3;
      it.dA = w + 3 * n3;
      it.dB = w + 4 * n3;
      it.dP = w + 5 * n3;
      it.tau0 = (float)tau0[base + t];
    }
    const dim3 grid(blocks, nb);
    const int tiles_i = (M + kF3TileI - 1) / kF3TileI, tiles_j = (M + kF3TileJ - 1) / kF3TileJ;
    const dim3 sgrid((unsigned)(tiles_i * tiles_j), (unsigned)((M + kF3PlanesPerBlock - 1) / kF3PlanesPerBlock),
                     (unsigned)nb);
    const dim3 sblock(kF3TileI, kF3TileJ);
    f3_phase_kernel<<<grid, kF3Threads, 0, s>>>(fb, F3_INIT, nsteps);
    int cur = 0;   // 0: the increment is in dA
    for (int step = 0; step < nsteps; ++step) {
      const int m = f3_sweeps(q, skew, step);   // >= 2
      for (int sw = 0; sw < m; ++sw) {
        const int face_step = step + 1 < nsteps ? step + 1 : -1;
        if (sw == 0)
          f3_sweep_kernel<F3S_FIRST><<<sgrid, sblock, 0, s>>>(fb, cur, tiles_i, face_step, step + 1 >= kF3ExtrapStart);
        else if (sw == m - 1)
          f3_sweep_kernel<F3S_LAST><<<sgrid, sblock, 0, s>>>(fb, cur, tiles_i, face_step, step + 1 >= kF3ExtrapStart);
        else
          f3_sweep_kernel<0><<<sgrid, sblock, 0, s>>>(fb, cur, tiles_i, face_step, step + 1 >= kF3ExtrapStart);
        cur ^= 1;
      }
    }
    f3_phase_kernel<<<grid, kF3Threads, 0, s>>>(fb, F3_OUT, nsteps);
    BS_CUDA_TRY(cudaGetLastError());
    BS_CUDA_TRY(cudaFreeAsync(ws, s));
  }
  return BS_OK;
}

}  // extern "C"
