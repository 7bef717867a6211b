// Three-asset operator (eq. bse_general with n = 3): the 19-point stencil and far-face
// data shared by the three-asset kernels (fine3.cu, krylov3.cu).  Layout u[(k*M + j)*M + i],
// i the index of asset 1; coefficients are host-rounded FP32 constants times exact integer
// node indices (x_p = i_p h, h cancels).
#pragma once

#include "common.cuh"

namespace bsp {

constexpr int kF3MaxItems = 32;
constexpr int kF3Threads = 256;
constexpr int kF3TileI = 32, kF3TileJ = 8;   // sweep kernel: columns per block
constexpr int kF3PlanesPerBlock = 8;         // sweep kernel: planes of k per thread

struct F3Item {
  const float* in;
  float* out;
  float* hi;   // [M^3] state, high part
  float* lo;   // [M^3] compensation
  float* b;    // [M^3] dtau R_h u of the step
  float* dA;   // [M^3] increment ping-pong
  float* dB;
  float* dP;   // [M^3] the previous step's increment
  float tau0;
};

struct F3Coef {
  float A[3];      // 1/2 sigma_p^2 dtau      (times i_p^2: diffusion weight of +-1 along p)
  float D[3];      // 1/2 r dtau              (times i_p: drift weight, + on +1, - on -1)
  float Cxy, Cxz, Cyz;   // 1/4 rho_pq sigma_p sigma_q dtau (times i_p i_q: cross weight)
  float rdt;       // r dtau
};

struct F3Batch {
  F3Item it[kF3MaxItems];
  int n, M;
  float h;
  F3Coef c;
  int kind;        // BS_PAYOFF_BASKET or BS_PAYOFF_EXCHANGE
  float w[3], K;   // basket: max(w.x - K e^{-r tau}, 0) on the far faces
  PayoffF ex;      // exchange: Margrabe in (x_1, x_2) on the far faces
  float r;
  float dtau;
};

__device__ __forceinline__ void f3_node(int e, int M, int& i, int& j, int& k) {
  const int MM = M * M;
  k = e / MM;
  const int rem = e - k * MM;
  j = rem / M;
  i = rem - j * M;
}

__device__ __forceinline__ float f3_far_field(const F3Batch& fb, int i, int j, int k, float tau) {
  const float x = i * fb.h, y = j * fb.h, z = k * fb.h;
  if (fb.kind == BS_PAYOFF_BASKET)
    return fmaxf(fb.w[0] * x + fb.w[1] * y + fb.w[2] * z - fb.K * expf(-fb.r * tau), 0.0f);
  return far_field(fb.ex, x, y, tau);
}

// Off-diagonal part of dtau R_h at the node of index L of a shared-memory tile with HI entries
// along i and HJ along j (column coefficients precomputed; no guards: a neighbour at index -1 is
// 0 in the tile and has weight 0).
struct F3Col {
  float wxp, wxm, wyp, wym, cxy, cxz, cyz;
};
template <int HI, int HJ>
__device__ __forceinline__ float f3_tile_offdiag(const float* t, int L, const F3Col& w, float az, float mz, float fk) {
  constexpr int X = 1, Y = HI, Z = HI * HJ;
  float acc = w.wxp * t[L + X];
  acc = fmaf(w.wxm, t[L - X], acc);
  acc = fmaf(w.wyp, t[L + Y], acc);
  acc = fmaf(w.wym, t[L - Y], acc);
  acc = fmaf(az + mz, t[L + Z], acc);
  acc = fmaf(az - mz, t[L - Z], acc);
  acc = fmaf(w.cxy, (t[L + X + Y] + t[L - X - Y]) - (t[L + X - Y] + t[L - X + Y]), acc);
  acc = fmaf(w.cxz * fk, (t[L + X + Z] + t[L - X - Z]) - (t[L + X - Z] + t[L - X + Z]), acc);
  acc = fmaf(w.cyz * fk, (t[L + Y + Z] + t[L - Y - Z]) - (t[L + Y - Z] + t[L - Y + Z]), acc);
  return acc;
}

// host helpers (fine3.cu)
int f3_check(int M, double xmax, const bs_params3* p);                 // BS_OK or BS_ERR_ARG
F3Batch f3_batch(int M, double xmax, const bs_params3& p, double dtau);  // coefficients of one step
double f3_contraction(int M, const bs_params3& p, double dtau);         // Gershgorin bound q
// G over one slice for one state, BiCGSTAB per implicit step (krylov3.cu)
size_t k3_workspace_bytes(int M);
int* k3_status(void* ws, int M);                                     // device int, zeroed by the caller
int coarse_propagate3_krylov(int M, double xmax, const bs_params3& p, const float* u_in, float* u_out, double tau0,
                             double dtau, int nsteps, double tol, int maxit, void* ws, cudaStream_t s);
int k3_result(void* ws, int M, int maxit, cudaStream_t s);           // synchronous

}  // namespace bsp
