// What the PINO's two network paths share: the state descriptor, the bilinear sample, and the
// interface of the cluster path (pino_cluster.cu).
#pragma once

#include "common.cuh"
#include "umma.cuh"

namespace bsp {

struct PinoState {
  const float* in;     // state grid u
  float* out;          // PROP: state grid result
  int M;
  float h;             // spacing of the state grid
  float tau, dtau;     // network time inputs
  float s1, s2, rho, r;
  PayoffF pf;
};

// The states of a launch: a device array, or (list NULL) one state in the launch's own parameters,
// which needs no copy ahead of it (one 128 x 128 state 47.1 -> 45.1 us).
struct PinoStates {
  const PinoState* list;
  PinoState one;
};

// bilinear sample of a node field on an Mi grid at fractional node index (ti, tj)
__device__ __forceinline__ float bilinear(const float* u, int Mi, float tx, float ty) {
  int i0 = min((int)floorf(tx), Mi - 2), j0 = min((int)floorf(ty), Mi - 2);
  i0 = max(i0, 0);
  j0 = max(j0, 0);
  const float fx = tx - i0, fy = ty - j0;
  const float* r0 = u + (size_t)j0 * Mi;
  const float* r1 = r0 + Mi;
  const float a = r0[i0] * (1.f - fx) + r0[i0 + 1] * fx;
  const float c = r1[i0] * (1.f - fx) + r1[i0 + 1] * fx;
  return a * (1.f - fy) + c * fy;
}

// Operands of the cluster path, laid out once as the shared-memory images it copies in.
struct PinoClusterNet {
  const float *lift_w, *lift_b, *pw_b, *b1, *w2;
  const bf16* dft_x;   // inverse x-DFT [128 x][32] (columns 24..26 one) then x-DFT [32][128 x], canonical
  const bf16* ey;      // y-DFT [48][256], canonical
  const bf16* eyi;     // inverse y-DFT [256][48], canonical
  const bf16* pw;      // [L][32][32] canonical (o, c)
  const bf16* w1;      // [H][32] canonical
  const bf16* mix;     // [L][72][2][4][4][32][4][2]: mode matrices, see pino_mix_index
  float b2;
  int L, H;
};

// Element (c -> o, re/im) of layer l's matrix of mode (q, kx) in PinoClusterNet::mix.  A unit is
// four consecutive q at one kx; a lane holds four outputs and four inputs of a half unit.
__host__ __device__ inline size_t pino_mix_index(int l, int q, int kx, int c, int o, int ri) {
  const int unit = (q >> 2) * 12 + kx, lane = (c >> 2) * 4 + ((o & 15) >> 2);
  return ((((((size_t)l * 72 + unit) * 2 + (o >> 4)) * 4 + (q & 3)) * 4 + (c & 3)) * 32 + lane) * 8 +
         (size_t)(o & 3) * 2 + ri;
}

// The network on B states (128 x 128 network grid): wout[b][y][x], the increment.
int launch_pino_cluster(const PinoClusterNet& net, const PinoStates& st, float* wout, int B, int* err,
                        cudaStream_t s);

}  // namespace bsp
