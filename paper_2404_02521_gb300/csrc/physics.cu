// PDE term of the PINO training loss (Sec. 3.5, eq. bs_totalloss) on the device.
//
// A coarse-propagator prediction u~ of u(tau + dtau) from u(tau) is scored by the residual of
// eq. (bse_change_variable), discretised by eq. (fd) with the slice as one implicit step, at
// the collocation points that carry a PDE row (0 <= i, j <= M-2):
//   r = (u~ - u_prev) / dtau - R_h u~ = ((u~ - u_prev) - dtau R_h u~) / dtau,
//   loss = (1/n) sum r^2  (n = (M-1)^2),   d loss / d u~_i = (2/n) sum_j r_j d r_j / d u~_i.
// Row j of R_h reads the 3 x 3 nodes around j, so the gradient at node i gathers the residuals
// of the (up to) nine collocation points around i from a tile in shared memory; no scratch
// plane is needed.  The residual is evaluated in FP32 from the same index-unit coefficients as the
// steppers (dtau R_h with the slice's dtau), the loss accumulated in FP64.
#include "common.cuh"

namespace bsp {

namespace {

struct PhysItem {
  const float* pred;
  const float* prev;
  float* grad;     // nullptr: loss only
  double* loss;    // device
  ItemDesc d;      // coefficients of dtau R_h
  float rdtau;     // 1 / dtau
};

constexpr int kPhysMaxItems = 32;
constexpr int kPhysThreads = 256;
constexpr size_t kPhysWideBlocks = 304;   // two blocks of the wide tile on every SM

struct PhysBatch {
  PhysItem it[kPhysMaxItems];
  int M;
  double inv_n;
};

// One block scores a tile of kPhysTile x kPhysTile nodes of one sample: the prediction is staged
// with two nodes around the tile, the residuals are formed once on the tile and one node around
// it, and the gradient gathers the nine around each node from shared memory.  Bound by the FP64
// sum of r^2 and the latency of the three phases.  Recomputing the nine residuals at every node
// from global memory, with an FP64 butterfly in every warp, took 21.1 us on the device for 32
// samples of 128 x 128 (now 12.6) and 36 us for 4 of 512 x 512 (15.3).
template <int kPhysTile>
__global__ void __launch_bounds__(kPhysThreads) physics_loss_kernel(const __grid_constant__ PhysBatch pb) {
  constexpr int kPhysP = kPhysTile + 4, kPhysR = kPhysTile + 2;
  const PhysItem& it = pb.it[blockIdx.y];
  const int M = pb.M, tid = threadIdx.x;
  const int tiles = (M + kPhysTile - 1) / kPhysTile;
  const int ty = blockIdx.x / tiles, i0 = (blockIdx.x - ty * tiles) * kPhysTile, j0 = ty * kPhysTile;
  __shared__ float u[kPhysP * kPhysP], r[kPhysR * kPhysR];
  for (int e = tid; e < kPhysP * kPhysP; e += kPhysThreads) {
    const int row = e / kPhysP, c = e - row * kPhysP, i = i0 + c - 2, j = j0 + row - 2;
    u[e] = i >= 0 && i < M && j >= 0 && j < M ? it.pred[j * M + i] : 0.f;
  }
  __syncthreads();
  // r at the collocation points; a neighbour at index -1 has weight 0, its entry is the point's own
  double r2 = 0.0;
  for (int e = tid; e < kPhysR * kPhysR; e += kPhysThreads) {
    const int row = e / kPhysR, c = e - row * kPhysR, i = i0 + c - 1, j = j0 + row - 1;
    float res = 0.f;
    if (i >= 0 && j >= 0 && i <= M - 2 && j <= M - 2) {
      float ce, cw, cgi, cs, cn, gj;
      column_coefs(it.d, i, ce, cw, cgi);
      row_coefs(it.d, j, cs, cn, gj);
      const float* y = u + (row + 1) * kPhysP + c + 1;
      const int w = i > 0 ? -1 : 0, n = j > 0 ? -kPhysP : 0;
      const float nW = y[n + w], nC = y[n], nE = y[n + 1], cW = y[w], cC = y[0], cE = y[1];
      const float sW = y[kPhysP + w], sC = y[kPhysP], sE = y[kPhysP + 1];
      // dtau R_h u~ (eq. fd in index units)
      const float t = ce * (cE - cC) - cw * (cC - cW) + cs * (sC - cC) - cn * (cC - nC) +
                      (cgi * gj) * ((sE - nE) - (sW - nW)) - it.d.rdt * cC;
      res = ((cC - it.prev[j * M + i]) - t) * it.rdtau;
      if (c >= 1 && c <= kPhysTile && row >= 1 && row <= kPhysTile) r2 += (double)res * (double)res;
    }
    r[e] = res;
  }
  __syncthreads();
  if (it.grad) {
    // d r_q / d u~_node = (delta - w_q(node - q)) / dtau over the collocation points q around the
    // node, w_q(o) the weight with which row q of dtau R_h reads its neighbour at offset o
    for (int e = tid; e < kPhysTile * kPhysTile; e += kPhysThreads) {
      const int row = e / kPhysTile, c = e % kPhysTile, i = i0 + c, j = j0 + row;
      if (i >= M || j >= M) continue;
      const float* y = r + (row + 1) * kPhysR + c + 1;
      float acc = 0.f;
      float ce[3], cw[3], cg[3], cs[3], cn[3], gj[3];   // of the columns i-1..i+1 and rows j-1..j+1
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        column_coefs(it.d, i + o - 1, ce[o], cw[o], cg[o]);
        row_coefs(it.d, j + o - 1, cs[o], cn[o], gj[o]);
      }
      // r is 0 at points outside the collocation set
#pragma unroll
      for (int dj = -1; dj <= 1; ++dj) {
#pragma unroll
        for (int di = -1; di <= 1; ++di) {
          const int qc = 1 - di, qr = 1 - dj;   // the node is q's neighbour at (di, dj)
          const float rq = y[-dj * kPhysR - di];
          float w;
          if (di == 0 && dj == 0) w = -(ce[qc] + cw[qc] + cs[qr] + cn[qr] + it.d.rdt);
          else if (dj == 0) w = di > 0 ? ce[qc] : cw[qc];
          else if (di == 0) w = dj > 0 ? cs[qr] : cn[qr];
          else w = di == dj ? cg[qc] * gj[qr] : -(cg[qc] * gj[qr]);
          acc = fmaf(rq, ((di == 0 && dj == 0) ? 1.f : 0.f) - w, acc);
        }
      }
      it.grad[j * M + i] = (float)(2.0 * pb.inv_n) * acc * it.rdtau;
    }
  }
  // block sum of r^2 (FP64), one atomic per block.  One warp folds the threads' sums from shared
  // memory: a butterfly in every warp is three times the FP64 instructions.
  __shared__ double part[kPhysThreads];
  part[tid] = r2;
  __syncthreads();
  if (tid >= 32) return;
  double s = part[tid];
#pragma unroll
  for (int w = 1; w < kPhysThreads / 32; ++w) s += part[tid + 32 * w];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (tid == 0 && s != 0.0) atomicAdd(it.loss, s * pb.inv_n);
}

}  // namespace

int launch_physics_loss(const bs_grid* g, const bs_params* p, const float* const* u_pred,
                        const float* const* u_prev, const double* dtau, int B, double* loss,
                        float* const* grad, cudaStream_t s) {
  const int M = g->M;
  PhysBatch pb;
  pb.M = M;
  pb.inv_n = 1.0 / ((double)(M - 1) * (double)(M - 1));
  BS_CUDA_TRY(cudaMemsetAsync(loss, 0, sizeof(double) * (size_t)B, s));
  for (int base = 0; base < B; base += kPhysMaxItems) {
    const int nb = B - base < kPhysMaxItems ? B - base : kPhysMaxItems;
    for (int k = 0; k < nb; ++k) {
      const int b = base + k;
      PhysItem& it = pb.it[k];
      it.pred = u_pred[b];
      it.prev = u_prev[b];
      it.grad = grad ? grad[b] : nullptr;
      it.loss = loss + b;
      it.d = make_item(p[b], 0.0, dtau[b]);
      it.rdtau = (float)(1.0 / dtau[b]);
    }
    // wide tiles recompute fewer residuals, narrow ones put more blocks on a chip that is not full
    // (device time, 32 / 16 nodes: 32 of 128 x 128 12.6 / 14.7 us, 4 of 512 x 512 15.3 / 22.2;
    // 8 of 128 x 128 8.8 / 8.5, 1 of 256 x 256 8.6 / 7.4, 4 of 64 x 64 8.4 / 6.4)
    const unsigned t32 = (unsigned)(M + 31) / 32, t16 = (unsigned)(M + 15) / 16;
    if ((size_t)t32 * t32 * nb >= kPhysWideBlocks)
      physics_loss_kernel<32><<<dim3(t32 * t32, (unsigned)nb), kPhysThreads, 0, s>>>(pb);
    else
      physics_loss_kernel<16><<<dim3(t16 * t16, (unsigned)nb), kPhysThreads, 0, s>>>(pb);
    BS_CUDA_TRY(cudaGetLastError());
  }
  return BS_OK;
}

}  // namespace bsp
