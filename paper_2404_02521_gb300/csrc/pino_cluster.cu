// K3 at 128 x 128: the whole PINO forward pass of one state as one cluster of CTAs.
//
// A state's activations (128 x 128 nodes, 32 channels, BF16: 1 MB) stay in the shared memory of
// the cluster, 128/CL rows of nodes per CTA, from the lifting to the projection; only the input
// state is read from and the increment written to global memory.  Per layer, with the rounding
// points of the staged path (BF16 operands, FP32 accumulation; umma.cuh):
//   G1  x-DFT of the CTA's rows: A = the activations of four rows as [(row, c)][x] (M-major, the
//       storage that G5 reads as [x][c]), B = the transform            -> X1 (c, kx, y, re/im)
//   --  all-to-all: a CTA gets 32/CL channels of every row (one bulk copy per pair of CTAs)
//   G2  y-DFT: A = X1 [(kx, c)][(y, re/im)], B = the transform         -> X2 (c, mode)
//   --  all-to-all: a CTA gets all channels of its 288/CL modes (asynchronous stores)
//   G3  mixing on the CUDA cores: one state per cluster makes it a matrix-vector product per
//       mode, whose weights (1.2 MB per layer) are read once per state -> Y (o, mode)
//   --  all-gather of Y (one bulk copy per pair of CTAs)
//   G4  inverse y-DFT of the CTA's own rows: A = Y [(kx, o)][(q, re/im)] -> Z1 (o, kx) per row
//   G5  inverse x-DFT + pointwise product into one accumulator per row; epilogue bias + ReLU
// then the projection, whose epilogue is the hidden layer's ReLU and dot product.
//
// Why: as one launch per stage and 128 x N tile, a batch of 128 states took 2247 us (21
// launches, activations through L2, 16k tiles of one MMA each per stage and scattered 2-byte
// stores) and one state 170 us, nearly all of it launch and tile latency.  Here the tensor work
// of a stage is a few dozen MMAs per CTA and the bound is the chain of stages: their epilogues and
// three exchanges per layer: one state 55 us, 128 states 625 us (with the apply kernel).
//
// An exchange needs no cluster barrier: the receiver's mbarrier counts the bytes, and a buffer
// is rewritten only after a later exchange has proved that its readers are done (Y/Z/stage
// share one region, the y-DFT and the x-DFT matrices another; the order is given at each).
// Every wait is bounded; a CTA whose wait ran out records the error, stops waiting and still
// takes part in the barriers.
#include "cluster_async.cuh"
#include "pino.cuh"

namespace bsp {

namespace {

constexpr int kPcThreads = 512;   // four sets of four warps; warp w % 4 reads TMEM lanes 32 (w % 4) ..

template <int CL>
struct PcCfg {
  static constexpr int ROWS = 128 / CL;     // rows of nodes per CTA
  static constexpr int G = ROWS / 4;        // groups of four rows
  static constexpr int CH = 32 / CL;        // channels per CTA in G2
  static constexpr int XCH = ROWS * 1536 / CL;   // bytes of X1 from one CTA to another
  static constexpr int XST = XCH + 64;      // their stride while staged (spreads the banks)
  static constexpr int HU = 144 / CL;       // half units (four modes, 16 outputs) per CTA in G3
  static constexpr int NU = (HU + 1) / 2;   // units whose inputs a CTA needs
  // shared memory
  static constexpr int ACT = 0;                       // [G][x / 8][row][c / 8][x % 8][c % 8]
  static constexpr int YZ = ACT + G * 32768;          // stage of X1, then Y, then Z1
  static constexpr int EA = YZ + 36864;               // x-DFTs, pointwise, inverse y-DFT | y-DFT | projection
  static constexpr int EA_PW = EA + 16384, EA_EYI = EA + 18432;
  static constexpr int RECV = EA + 24576;             // X1 [source][(kx, c) / 8][y / 4][row % 8][16 B]
  static constexpr int YST = RECV + ROWS * 1536;      // this CTA's part of Y
  static constexpr int X2 = YST + HU * 256;           // [unit][q][c] (re, im)
  static constexpr int FLT = X2 + NU * 512;           // lifting [4][32], bias [32], b1 [256], w2 [256]
  static constexpr int BAR = FLT + 4 * (128 + 32 + 512);
  static constexpr int SMEM = BAR + 192;
  static_assert(CL * XST <= 36864 && ROWS * 2048 <= 36864 && SMEM <= 232448, "shared memory");
  // G2 reads 128 rows of A and uses 12 CH of them: the rest lies within shared memory
  static_assert(RECV + (CL - 1) * XCH + (G / 2 - 1) * 256 + 16 * G * 128 <= SMEM, "rows beyond X1");
};

struct PcBars {
  uint64_t g1[4], g5[4], pr[4], g2, g4, x1, x2, y, lda, ldy;
};
static_assert(sizeof(PcBars) <= 176, "barriers");

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* mb) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_addr(mb))
               : "memory");
}
__device__ __forceinline__ void bulk_s2c(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t mb) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "r"(src), "r"(bytes), "r"(mb)
               : "memory");
}
__device__ __forceinline__ void st_async_u32(uint32_t dst, uint32_t v, uint32_t mb) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];\n" ::"r"(dst), "r"(v), "r"(mb)
               : "memory");
}

// one MMA of 128 x N x 16; a_mn: A is M-major
__device__ __forceinline__ void pc_mma(uint32_t d, uint64_t a, uint64_t b, int N, bool a_mn, bool acc) {
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) |
                         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
               " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1u : 0u));
}

// N consecutive accumulator columns of this warp's 32 lanes
template <int N>
__device__ __forceinline__ void pc_ld(uint32_t addr, uint32_t (&r)[N]) {
  static_assert(N == 4 || N == 8 || N == 16, "columns");
  if constexpr (N == 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
  } else if constexpr (N == 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(addr));
  }
}
__device__ __forceinline__ void pc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

template <int CL>
__global__ void __launch_bounds__(kPcThreads, 1)
pino_cluster_kernel(const __grid_constant__ PinoClusterNet net, const PinoState* __restrict__ st,
                    float* __restrict__ wout, int* err) {
  using F = PcCfg<CL>;
  constexpr int G = F::G, ROWS = F::ROWS;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sm = smem_addr(smem);
  PcBars& bar = *reinterpret_cast<PcBars*>(smem + F::BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + F::BAR + 176);
  float* flift = reinterpret_cast<float*>(smem + F::FLT);
  float* fbias = flift + 128;
  float* fb1 = fbias + 32;
  float* fw2 = fb1 + 256;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, set = warp >> 2, quad = warp & 3;
  const int rank = blockIdx.x, b = blockIdx.y, y0 = rank * ROWS;
  const PinoState s = st[b];
  bool ok = true;
  auto wait1 = [&](uint64_t* mb, uint32_t parity) {   // one thread
    if (ok && !mbar_wait(mb, parity)) {
      ok = false;
      atomicExch(err, 1);
    }
  };
  auto wait = [&](uint64_t* mb, uint32_t parity) {    // a whole warp
    wait1(mb, parity);
    __syncwarp();
  };

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    uint64_t* all = reinterpret_cast<uint64_t*>(&bar);
    for (int k = 0; k < (int)(sizeof(PcBars) / 8); ++k) mbar_init(all + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n");
    mbar_arm(&bar.lda, 16384);
    bulk_g2s(sm + F::EA, net.dft_x, 16384, &bar.lda);
    mbar_arm(&bar.x1, ROWS * 1536);
    mbar_arm(&bar.x2, F::NU * 512);
    mbar_arm(&bar.y, 36864);
  }
  // the lifting's parts that are the same at every node
  if (tid >= 32 && tid < 64) {
    const int o = lane;
    const float a[6] = {s.tau, s.dtau, s.s1, s.s2, s.rho, s.r};
    float v = net.lift_b[o];
#pragma unroll
    for (int c = 0; c < 6; ++c) v = fmaf(a[c], net.lift_w[(3 + c) * 32 + o], v);
    flift[o] = v;
#pragma unroll
    for (int c = 0; c < 3; ++c) flift[32 * (c + 1) + o] = net.lift_w[c * 32 + o];
  }
  for (int k = tid; k < net.H; k += kPcThreads) {
    fb1[k] = net.b1[k];
    fw2[k] = net.w2[k];
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = *tslot;
  const uint32_t tlane = tmem + ((uint32_t)(quad * 32) << 16);
  cluster_arrive();   // the barriers of every CTA exist before the first exchange

  // this thread's node column, and where its 16 bytes of channels 8 cc .. of row 4 g + set lie
  const int px = quad * 32 + lane;
  unsigned char* act_px = smem + F::ACT + (px >> 3) * 2048 + set * 512 + (px & 7) * 16;
  {
    const float hp = s.h * (float)(s.M - 1) / 127.f;   // network grid spacing
    const float ratio = (float)(s.M - 1) / 127.f;
    float u[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int y = y0 + 4 * g + set;
      u[g] = s.M == 128 ? s.in[y * 128 + px] : bilinear(s.in, s.M, px * ratio, y * ratio);
    }
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
      float base[8], wu[8], wy[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int o = cc * 8 + k;
        base[k] = fmaf(px * hp, flift[64 + o], flift[o]);
        wu[k] = flift[32 + o];
        wy[k] = flift[96 + o];
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float y = (float)(y0 + 4 * g + set) * hp;
        uint32_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          h[k] = pack_bf16(fmaf(u[g], wu[2 * k], fmaf(y, wy[2 * k], base[2 * k])),
                           fmaf(u[g], wu[2 * k + 1], fmaf(y, wy[2 * k + 1], base[2 * k + 1])));
        *reinterpret_cast<uint4*>(act_px + g * 32768 + cc * 128) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
  }

  // G1 of group g: D[(row, c)][(kx, re/im)] in the columns of the group's first row
  auto issue_g1 = [&](int g) {
#pragma unroll 1
    for (int kk = 0; kk < 8; ++kk)
      pc_mma(tmem + g * 128, umma_desc(sm + F::ACT + g * 32768 + kk * 4096, 2048, 128),
             umma_desc(sm + F::EA + 8192 + kk * 256, 128, 2048), 32, true, kk > 0);
    umma_commit(&bar.g1[g]);
  };
  proxy_fence();
  tc_before();
  __syncthreads();
  cluster_wait();
  if (tid == 0) {
    tc_after();
    wait1(&bar.lda, 0);
    for (int g = 0; g < G; ++g) issue_g1(g);
  }
  __syncwarp();

#pragma unroll 1
  for (int l = 0; l < net.L; ++l) {
    const uint32_t par = l & 1;
    // ---- X1: lane = c, quad = row of the group; a value goes to the CTA that owns channel c
    {
      constexpr int HV = G == 4 ? 2 : 1;   // halves of kx per thread
      const int g = set % G;
      wait(&bar.g1[g], par);
      tc_after();
      const int dst = lane / F::CH, cl = lane % F::CH;
      uint32_t v[HV][16];
#pragma unroll
      for (int hv = 0; hv < HV; ++hv) {
        const int kx0 = HV == 2 ? 6 * hv : 6 * (set / G);
        pc_ld<16>(tlane + g * 128 + 2 * kx0, v[hv]);
      }
      pc_ld_wait();
#pragma unroll
      for (int hv = 0; hv < HV; ++hv) {
        const int kx0 = HV == 2 ? 6 * hv : 6 * (set / G);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const int row = (kx0 + k) * F::CH + cl;
          *reinterpret_cast<uint32_t*>(smem + F::YZ + dst * F::XST + (row >> 3) * (G * 128) + g * 128 + (row & 7) * 16 +
                                       quad * 4) =
              pack_bf16(__uint_as_float(v[hv][2 * k]), __uint_as_float(v[hv][2 * k + 1]));
        }
      }
    }
    if (tid < 32) fbias[tid] = net.pw_b[l * 32 + tid];
    proxy_fence();
    tc_before();
    __syncthreads();
    if (warp == 0) {
      // every G1 is complete: the x-DFT's region takes the y-DFT
      if (lane == 0) {
        mbar_arm(&bar.ldy, 24576);
        bulk_g2s(sm + F::EA, net.ey, 24576, &bar.ldy);
      }
      if (lane < CL)
        bulk_s2c(cluster_addr(sm + F::RECV + rank * F::XCH, lane), sm + F::YZ + lane * F::XST, F::XCH,
                 cluster_addr(smem_addr(&bar.x1), lane));
      // ---- G2
      if (lane == 0) {
        wait1(&bar.ldy, par);
        wait1(&bar.x1, par);
        mbar_arm(&bar.x1, ROWS * 1536);
        tc_after();
#pragma unroll 1
        for (int k = 0; k < 16; ++k) {
          const int src = k / (G / 2), ks = k % (G / 2);
          pc_mma(tmem, umma_desc(sm + F::RECV + src * F::XCH + ks * 256, 128, G * 128),
                 umma_desc(sm + F::EA + k * 256, 128, 4096), 48, false, k > 0);
        }
        umma_commit(&bar.g2);
      }
      __syncwarp();
    }
    // the first mode matrices of G3, in flight meanwhile
    const bf16* mix = net.mix + (size_t)l * (72 * 2 * 4 * 1024) + lane * 8;
    uint4 wv[4];
    auto load_mix = [&](int task) {
      const uint4* p = reinterpret_cast<const uint4*>(mix + ((size_t)(rank * F::HU + (task >> 2)) * 4 + (task & 3)) * 1024);
#pragma unroll
      for (int j = 0; j < 4; ++j) wv[j] = __ldg(p + 32 * j);
    };
    load_mix(warp);
    // ---- X2: lane = (kx, c), columns (q, re/im); a value goes to the CTA(s) that mix its mode
    wait(&bar.g2, par);
    tc_after();
    if (tid == 0) {
      // G2 has read the y-DFT: its region takes back the x-DFTs, and the layer's other operands
      constexpr uint32_t kEyi = ROWS * 2 * 96;
      mbar_arm(&bar.lda, 16384 + 2048 + kEyi);
      bulk_g2s(sm + F::EA, net.dft_x, 16384, &bar.lda);
      bulk_g2s(sm + F::EA_PW, net.pw + (size_t)l * 1024, 2048, &bar.lda);
      bulk_g2s(sm + F::EA_EYI, net.eyi + (size_t)rank * (kEyi / 2), kEyi, &bar.lda);
    }
    __syncwarp();
    if (quad * 32 < 12 * F::CH) {
      const int row = quad * 32 + lane;
      uint32_t v[16];
      pc_ld<16>(tlane + set * 12, v);
      pc_ld_wait();
      if (row < 12 * F::CH) {
        const int kx = row / F::CH, c = rank * F::CH + row % F::CH;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const int q = set * 6 + k, unit = (q >> 2) * 12 + kx;
          const uint32_t val = pack_bf16(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1]));
          const int o0 = 2 * unit / F::HU, o1 = (2 * unit + 1) / F::HU;
          auto send = [&](int to) {
            st_async_u32(cluster_addr(sm + F::X2 + ((unit - to * F::HU / 2) * 4 + (q & 3)) * 128 + c * 4, to), val,
                         cluster_addr(smem_addr(&bar.x2), to));
          };
          send(o0);
          if (o1 != o0) send(o1);
        }
      }
    }
    // ---- G3: a warp per (half unit, q); lane = output o % 16 and half of the inputs
    wait(&bar.x2, par);
    if (tid == 0) mbar_arm(&bar.x2, F::NU * 512);
    __syncwarp();
#pragma unroll 1
    for (int task = warp; task < 4 * F::HU; task += kPcThreads / 32) {
      const int hu = task >> 2, q = task & 3, unit = (rank * F::HU + hu) >> 1, u0 = rank * F::HU / 2;
      uint4 w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = wv[j];
      if (task + kPcThreads / 32 < 4 * F::HU) load_mix(task + kPcThreads / 32);
      const uint4* xp = reinterpret_cast<const uint4*>(smem + F::X2 + ((unit - u0) * 4 + q) * 128 + (lane >> 4) * 64);
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint4 xv = xp[j];
        const uint32_t xs[4] = {xv.x, xv.y, xv.z, xv.w}, ws[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float xr = bf_lo(xs[i]), xi = bf_hi(xs[i]), wr = bf_lo(ws[i]), wi = bf_hi(ws[i]);
          re = fmaf(-xi, wi, fmaf(xr, wr, re));
          im = fmaf(xi, wr, fmaf(xr, wi, im));
        }
      }
      re += __shfl_xor_sync(0xffffffffu, re, 16);
      im += __shfl_xor_sync(0xffffffffu, im, 16);
      if (lane < 16)
        *reinterpret_cast<uint32_t*>(smem + F::YST + hu * 256 + (lane >> 3) * 128 + (lane & 7) * 16 + q * 4) =
            pack_bf16(re, im);
    }
    proxy_fence();
    tc_before();
    __syncthreads();
    if (warp == 0) {
      if (lane < CL)
        bulk_s2c(cluster_addr(sm + F::YZ + rank * (F::HU * 256), lane), sm + F::YST, F::HU * 256,
                 cluster_addr(smem_addr(&bar.y), lane));
      // ---- G4
      if (lane == 0) {
        wait1(&bar.lda, (l + 1) & 1);
        wait1(&bar.y, par);
        mbar_arm(&bar.y, 36864);
        tc_after();
#pragma unroll 1
        for (int t = 0; t < 3; ++t)
#pragma unroll 1
          for (int kk = 0; kk < 3; ++kk)
            pc_mma(tmem + 64 + t * 32, umma_desc(sm + F::YZ + t * 2048 + kk * 12288, 6144, 128),
                   umma_desc(sm + F::EA_EYI + kk * 256, 128, 768), 2 * ROWS, false, kk > 0);
        umma_commit(&bar.g4);
      }
      __syncwarp();
    }
    // ---- Z1 over Y (every G4 is complete): lane = o, quad = kx % 4; set takes G of the rows
    wait(&bar.g4, par);
    tc_after();
    {
      uint32_t v[3][2 * G];
#pragma unroll
      for (int t = 0; t < 3; ++t) pc_ld<2 * G>(tlane + 64 + t * 32 + set * 2 * G, v[t]);
      pc_ld_wait();
      unsigned char* z = smem + F::YZ + (lane >> 3) * 512 + (lane & 7) * 16 + quad * 4;
#pragma unroll
      for (int t = 0; t < 3; ++t)
#pragma unroll
        for (int i = 0; i < G; ++i)
          *reinterpret_cast<uint32_t*>(z + (set * G + i) * 2048 + t * 128) =
              pack_bf16(__uint_as_float(v[t][2 * i]), __uint_as_float(v[t][2 * i + 1]));
      // K = 24 .. 31 is padding
      if (tid < ROWS * 32)
        *reinterpret_cast<uint4*>(smem + F::YZ + (tid >> 5) * 2048 + (lane >> 3) * 512 + 384 + (lane & 7) * 16) =
            make_uint4(0, 0, 0, 0);
    }
    proxy_fence();
    tc_before();
    __syncthreads();
    // ---- G5
    if (tid == 0) {
      tc_after();
#pragma unroll 1
      for (int g = 0; g < G; ++g) {
#pragma unroll 1
        for (int r = 0; r < 4; ++r) {
          const uint32_t d = tmem + (g * 4 + r) * 32;
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
            pc_mma(d, umma_desc(sm + F::EA + kk * 256, 128, 512),
                   umma_desc(sm + F::YZ + (g * 4 + r) * 2048 + kk * 256, 128, 512), 32, false, kk > 0);
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
            pc_mma(d, umma_desc(sm + F::ACT + g * 32768 + r * 512 + kk * 256, 128, 2048),
                   umma_desc(sm + F::EA_PW + kk * 256, 128, 512), 32, false, true);
        }
        umma_commit(&bar.g5[g]);
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      wait(&bar.g5[g], par);
      tc_after();
      uint32_t v[2][16];
      pc_ld<16>(tlane + (g * 4 + set) * 32, v[0]);
      pc_ld<16>(tlane + (g * 4 + set) * 32 + 16, v[1]);
      pc_ld_wait();
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        uint32_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int o = cc * 8 + 2 * k;
          h[k] = pack_bf16(fmaxf(__uint_as_float(v[o >> 4][o & 15]) + fbias[o], 0.f),
                           fmaxf(__uint_as_float(v[o >> 4][(o & 15) + 1]) + fbias[o + 1], 0.f));
        }
        *reinterpret_cast<uint4*>(act_px + g * 32768 + cc * 128) = make_uint4(h[0], h[1], h[2], h[3]);
      }
      proxy_fence();
      tc_before();
      __syncthreads();
      if (l + 1 < net.L) {
        if (tid == 0) {
          tc_after();
          issue_g1(g);
        }
        __syncwarp();
      }
    }
  }

  // ---- projection: set takes a row of each group, its first thread issues the row's products
  if (tid == 0) {
    mbar_arm(&bar.lda, net.H * 64);
    bulk_g2s(sm + F::EA, net.w1, net.H * 64, &bar.lda);
  }
  __syncwarp();
  wait(&bar.lda, (net.L + 1) & 1);
  uint32_t ppar = 0;
#pragma unroll 1
  for (int g = 0; g < G; ++g) {
    float acc = 0.f;
#pragma unroll 1
    for (int h0 = 0; h0 < net.H; h0 += 128) {
      const int n = min(128, net.H - h0);
      if (quad == 0 && lane == 0) {
        tc_after();
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
          pc_mma(tmem + set * 128, umma_desc(sm + F::ACT + g * 32768 + set * 512 + kk * 256, 128, 2048),
                 umma_desc(sm + F::EA + h0 * 64 + kk * 256, 128, 512), n, false, kk > 0);
        umma_commit(&bar.pr[set]);
      }
      __syncwarp();
      wait(&bar.pr[set], ppar);
      ppar ^= 1;
      tc_after();
#pragma unroll 1
      for (int c0 = 0; c0 < n; c0 += 16) {
        uint32_t v[16];
        pc_ld<16>(tlane + set * 128 + c0, v);
        pc_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k)
          acc = fmaf(fmaxf(__uint_as_float(v[k]) + fb1[h0 + c0 + k], 0.f), fw2[h0 + c0 + k], acc);
      }
      tc_before();
      asm volatile("bar.sync %0, 128;\n" ::"r"(1 + set) : "memory");
    }
    wout[((size_t)b * 128 + y0 + 4 * g + set) * 128 + px] = acc + net.b2;
  }
  tc_before();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
  // the copies that this CTA sent have been received before its shared memory goes away
  cluster_arrive();
  cluster_wait();
}

template <int CL>
cudaError_t pc_attributes() {
  cudaError_t e = cudaFuncSetAttribute(pino_cluster_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       PcCfg<CL>::SMEM);
  if (e == cudaSuccess && CL > 8)
    e = cudaFuncSetAttribute(pino_cluster_kernel<CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <int CL>
void pc_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int B, cudaStream_t s) {
  cfg = {};
  cfg.gridDim = dim3(CL, (unsigned)B, 1);
  cfg.blockDim = dim3(kPcThreads, 1, 1);
  cfg.dynamicSmemBytes = PcCfg<CL>::SMEM;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

// clusters that run at once (0 if the size cannot be launched)
template <int CL>
int pc_capacity() {
  static const int n = [] {
    int v = 0;
    if (pc_attributes<CL>() != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    pc_config<CL>(cfg, attr, 1, nullptr);
    return cudaOccupancyMaxActiveClusters(&v, pino_cluster_kernel<CL>, &cfg) == cudaSuccess ? v : 0;
  }();
  return n;
}

template <int CL>
int pc_launch(const PinoClusterNet& net, const PinoState* st, float* wout, int B, int* err, cudaStream_t s) {
  BS_CUDA_TRY(pc_attributes<CL>());
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  pc_config<CL>(cfg, attr, B, s);
  BS_CUDA_TRY(cudaLaunchKernelEx(&cfg, pino_cluster_kernel<CL>, net, st, wout, err));
  return BS_OK;
}

}  // namespace

int launch_pino_cluster(const PinoClusterNet& net, const PinoState* st, float* wout, int B, int* err,
                        cudaStream_t s) {
  // Clusters of 16 halve every stage's rows (one to seven states 56 us, against 76 with 8) while
  // they all run at once; beyond that twice as many clusters of 8 fit (8 states: 76 us, against
  // 112 in two waves of 16; 15 states 79).
  const int c16 = pc_capacity<16>(), c8 = pc_capacity<8>();
  if (c16 > 0 && (c8 == 0 || B <= c16)) return pc_launch<16>(net, st, wout, B, err, s);
  return pc_launch<8>(net, st, wout, B, err, s);
}

}  // namespace bsp
