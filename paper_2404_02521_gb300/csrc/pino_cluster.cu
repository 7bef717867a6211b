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
// three exchanges per layer: one state 45 us, 128 states 506 us (with the apply kernel).  Per layer at
// CL = 8 (22 k cycles): MMAs 7.5 k (a 128 x N x 16 MMA takes 64 cycles and more at N = 32, the A tile's
// fetch; the M-major ones 100), G3 3.6 k, exchanges 5 k, epilogues 4 k.
//
// An exchange needs no cluster barrier: the receiver's mbarrier counts the bytes, and a buffer
// is rewritten only after a later exchange has proved that its readers are done (Y/Z/stage
// share one region, the y-DFT and the x-DFT matrices another; the order is given at each).
// Every wait is bounded; a CTA whose wait ran out records the error, stops waiting and still
// takes part in the barriers.
#include <map>
#include <mutex>

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
  static constexpr int EA = YZ + 36864;               // y-DFT | inverse x-DFT, pointwise, inverse y-DFT
  static constexpr int EA_PW = EA + 8192, EA_EYI = EA + 10240;
  // RECV holds X1 until G2 has read it, then mode matrices, in the last layer then the projection
  static constexpr int RECV = EA + 24576;             // X1 [source][(kx, c) / 8][y / 4][row % 8][16 B]
  static constexpr int YST = RECV + (ROWS * 1536 > 16384 ? ROWS * 1536 : 16384);   // this CTA's part of Y
  static constexpr int X2 = YST + HU * 256;           // [unit][q][c] (re, im); outside G2 .. G3 the x-DFT
  static constexpr int FLT = X2 + 6144;               // lifting [4][32]
  // mode matrices of G3 tasks that wait in shared memory: all of the next layer's if there is
  // room, else 12 that follow the two per warp held in registers
  static constexpr bool MIX_ALL = CL == 16;
  static constexpr int MIX = MIX_ALL ? FLT + 512 : RECV;
  static constexpr int MIX_TASKS = MIX_ALL ? 4 * HU : 12;
  static_assert(NU * 512 <= 6144 && (MIX_ALL || MIX_TASKS * 2048 <= YST - RECV), "regions");
  static constexpr int BAR = FLT + 512 + (MIX_ALL ? MIX_TASKS * 2048 : 0);
  // (G1 reads 32 rows of the x-DFT and uses 24: the rest, too, lies within shared memory)
  static constexpr int SMEM = BAR + 192 > X2 + 8192 ? BAR + 192 : X2 + 8192;
  static_assert(CL * XST <= 36864 && ROWS * 2048 <= 36864 && SMEM <= 232448, "shared memory");
  // G2 reads 128 rows of A and uses 12 CH of them: the rest lies within shared memory
  static_assert(RECV + (CL - 1) * XCH + (G / 2 - 1) * 256 + 16 * G * 128 <= SMEM, "rows beyond X1");
};

struct PcBars {
  uint64_t g1[4], g5[4], pr[4], g2, g4, x1, x2, y, lda, ldy, ldx, ldm, ldw;
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

// A shared-memory operand descriptor in its two words; at(off) moves the start address.  Built
// once per operand: a descriptor assembled from its fields before each MMA made the issuing
// thread the bound (90 cycles per MMA; now an addition).
struct PcDesc {
  uint32_t lo, hi;
  __device__ __forceinline__ PcDesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    const uint64_t d = umma_desc(addr, lbo, sbo);
    lo = (uint32_t)d;
    hi = (uint32_t)(d >> 32);
  }
  __device__ __forceinline__ PcDesc at(uint32_t off) const {
    PcDesc d = *this;
    d.lo += off >> 4;
    return d;
  }
};

// one MMA of 128 x N x 16; A_MN: A is M-major
constexpr uint32_t pc_idesc(int N, bool a_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void pc_mma(uint32_t d, const PcDesc& a, const PcDesc& b, uint32_t idesc, bool acc) {
  asm volatile("{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %6, 0;\n mov.b64 da, {%1, %2};\n"
               " mov.b64 db, {%3, %4};\n tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n"
               ::"r"(d), "r"(a.lo), "r"(a.hi), "r"(b.lo), "r"(b.hi), "r"(idesc), "r"(acc ? 1u : 0u));
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

// a load of constant data that stays where it is written (ahead of a wait)
__device__ __forceinline__ uint4 ld_early(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// pairs of FP32 values, and the packed operations on them
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t relu_bf16(uint32_t v) {   // (NaN gives 0)
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&v), __float2bfloat162_rn(0.f));
  return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

template <int CL>
__global__ void __launch_bounds__(kPcThreads, 1)
pino_cluster_kernel(const __grid_constant__ PinoClusterNet net, const __grid_constant__ PinoStates st,
                    float* __restrict__ wout, int* err) {
  using F = PcCfg<CL>;
  constexpr int G = F::G, ROWS = F::ROWS;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sm = smem_addr(smem);
  PcBars& bar = *reinterpret_cast<PcBars*>(smem + F::BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + F::BAR + 176);
  float* flift = reinterpret_cast<float*>(smem + F::FLT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, set = warp >> 2, quad = warp & 3;
  const int rank = blockIdx.x, b = blockIdx.y, y0 = rank * ROWS;
  const bool leader = quad == 0 && lane == 0;   // of the set
  const PinoState s = st.list ? st.list[b] : st.one;
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

  // this thread's nodes: column px of the rows r0 .. r0 + G - 1 of the group grp; their values of
  // the state are in flight during the set-up.  The sets of a group need no others' progress
  // between the inverse transform and the next x-DFT.
  const int px = quad * 32 + lane, grp = set % G, r0 = set / G * G, yt = y0 + 4 * grp + r0;
  float u[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int y = yt + g;
    const float ratio = (float)(s.M - 1) / 127.f;
    u[g] = s.M == 128 ? s.in[y * 128 + px] : bilinear(s.in, s.M, px * ratio, y * ratio);
  }
  const bf16* mix = net.mix + (size_t)(rank * F::HU * 4) * 1024;
  auto load_mix_smem = [&](int l) {   // one thread
    mbar_arm(&bar.ldm, F::MIX_TASKS * 2048);
    bulk_g2s(sm + F::MIX, mix + ((size_t)l * 576 + (F::MIX_ALL ? 0 : 32)) * 1024, F::MIX_TASKS * 2048, &bar.ldm);
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    uint64_t* all = reinterpret_cast<uint64_t*>(&bar);
    for (int k = 0; k < (int)(sizeof(PcBars) / 8); ++k) mbar_init(all + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n");
    mbar_arm(&bar.ldx, 6144);
    bulk_g2s(sm + F::X2, net.dft_x + 4096, 6144, &bar.ldx);
    mbar_arm(&bar.ldy, 24576);
    bulk_g2s(sm + F::EA, net.ey, 24576, &bar.ldy);
    if (F::MIX_ALL) load_mix_smem(0);
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
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = *tslot;
  const uint32_t tlane = tmem + ((uint32_t)(quad * 32) << 16);
  cluster_arrive();   // the barriers of every CTA exist before the first exchange

  // where 16 bytes of channels 8 cc .. of this thread's nodes lie
  unsigned char* act_px = smem + F::ACT + grp * 32768 + (px >> 3) * 2048 + r0 * 512 + (px & 7) * 16;
  {
    const float hp = s.h * (float)(s.M - 1) / 127.f;   // network grid spacing
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
        const float y = (float)(yt + g) * hp;
        uint32_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          h[k] = pack_bf16(fmaf(u[g], wu[2 * k], fmaf(y, wy[2 * k], base[2 * k])),
                           fmaf(u[g], wu[2 * k + 1], fmaf(y, wy[2 * k + 1], base[2 * k + 1])));
        *reinterpret_cast<uint4*>(act_px + g * 512 + cc * 128) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
  }

  // G1 of group g: D[(row, c)][(kx, re/im)] in the columns of the group's first row
  auto issue_g1 = [&](int g) {
    const PcDesc a(sm + F::ACT + g * 32768, 2048, 128), x(sm + F::X2, 128, 2048);
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
      pc_mma(tmem + g * 128, a.at(kk * 4096), x.at(kk * 256), pc_idesc(32, true), kk > 0);
    umma_commit(&bar.g1[g]);
  };
  proxy_fence();
  tc_before();
  __syncthreads();
  cluster_wait();
  if (leader && set < G) {
    tc_after();
    wait1(&bar.ldx, 0);
    issue_g1(set);
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
      if (l > 0) {   // the stage takes the place of Z1
#pragma unroll
        for (int k = 0; k < G; ++k) wait(&bar.g5[k], par ^ 1);
      }
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
    proxy_fence();
    tc_before();
    __syncthreads();
    if (warp < CL && lane == 0)   // a copy per warp: one warp issuing them all took 1000 cycles
      bulk_s2c(cluster_addr(sm + F::RECV + rank * F::XCH, warp), sm + F::YZ + warp * F::XST, F::XCH,
               cluster_addr(smem_addr(&bar.x1), warp));
    __syncwarp();
    if (warp == 0) {
      // ---- G2
      if (lane == 0) {
        wait1(&bar.ldy, par);
        wait1(&bar.x1, par);
        mbar_arm(&bar.x1, ROWS * 1536);
        tc_after();
        const PcDesc a(sm + F::RECV, 128, G * 128), e(sm + F::EA, 128, 4096);
#pragma unroll
        for (int k = 0; k < 16; ++k)
          pc_mma(tmem, a.at(k / (G / 2) * F::XCH + k % (G / 2) * 256), e.at(k * 256), pc_idesc(48, false), k > 0);
        umma_commit(&bar.g2);
      }
      __syncwarp();
    }
    // the first mode matrices of G3, in flight meanwhile
    uint4 wa[4], wb[4];
    auto load_mix = [&](uint4 (&wv)[4], int task) {
      const uint4* p = reinterpret_cast<const uint4*>(mix + ((size_t)l * 576 + task) * 1024 + lane * 8);
#pragma unroll
      for (int j = 0; j < 4; ++j) wv[j] = ld_early(p + 32 * j);
    };
    if (!F::MIX_ALL) {
      load_mix(wa, warp);
      load_mix(wb, warp + 16);
    }
    // ---- X2: lane = (kx, c), columns (q, re/im); a value goes to the CTA(s) that mix its mode
    wait(&bar.g2, par);
    tc_after();
    if (tid == 0) {
      // G2 has read the y-DFT and X1: their regions take the operands of the stages that follow
      constexpr uint32_t kEyi = ROWS * 2 * 96;
      if (!F::MIX_ALL) load_mix_smem(l);
      mbar_arm(&bar.lda, 8192 + 2048 + kEyi);
      bulk_g2s(sm + F::EA, net.dft_x, 8192, &bar.lda);
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
    // ---- G3: a warp per (half unit, q); a lane multiplies 4 inputs into 4 outputs, so that its inputs
    // are one shared-memory read (a broadcast read per input and output pair made the return path to
    // the registers the bound: 4800 cycles at CL = 8)
    wait(&bar.x2, par);
    if (tid == 0) mbar_arm(&bar.x2, F::NU * 512);
    __syncwarp();
    auto mix_task = [&](uint4 (&wv)[4], int task, int next) {
      const int hu = task >> 2, q = task & 3, unit = (rank * F::HU + hu) >> 1, u0 = rank * F::HU / 2;
      const uint4 xv = *reinterpret_cast<const uint4*>(smem + F::X2 + ((unit - u0) * 4 + q) * 128 + (lane >> 2) * 16);
      const uint32_t xs[4] = {xv.x, xv.y, xv.z, xv.w};
      uint64_t br[4] = {0, 0, 0, 0}, bi[4] = {0, 0, 0, 0};   // the sums of re(x) (wr, wi) and of im(x) (wr, wi)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint64_t xr = pack2(bf_lo(xs[i]), bf_lo(xs[i])), xi = pack2(bf_hi(xs[i]), bf_hi(xs[i]));
        const uint32_t ws[4] = {wv[i].x, wv[i].y, wv[i].z, wv[i].w};
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const uint64_t w = pack2(bf_lo(ws[o]), bf_hi(ws[o]));
          br[o] = fma2(xr, w, br[o]);
          bi[o] = fma2(xi, w, bi[o]);
        }
      }
      if (next < 4 * F::HU) load_mix(wv, next);
      float re[4], im[4];
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        float rr, ri, ir, ii;
        unpack2(br[o], rr, ri);
        unpack2(bi[o], ir, ii);
        re[o] = rr - ii;
        im[o] = ri + ir;
      }
      // sum over the eight lanes of the same outputs, halving what a lane holds: lane bits 4 and 3
      // choose the output, bit 2 re or im
      const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const float sr = __shfl_xor_sync(0xffffffffu, h4 ? re[o] : re[o + 2], 16);
        const float si = __shfl_xor_sync(0xffffffffu, h4 ? im[o] : im[o + 2], 16);
        re[o] = (h4 ? re[o + 2] : re[o]) + sr;
        im[o] = (h4 ? im[o + 2] : im[o]) + si;
      }
      const float sr = __shfl_xor_sync(0xffffffffu, h3 ? re[0] : re[1], 8);
      const float si = __shfl_xor_sync(0xffffffffu, h3 ? im[0] : im[1], 8);
      const float r1 = (h3 ? re[1] : re[0]) + sr, i1 = (h3 ? im[1] : im[0]) + si;
      const float v = (h2 ? i1 : r1) + __shfl_xor_sync(0xffffffffu, h2 ? r1 : i1, 4);
      const float vi = __shfl_xor_sync(0xffffffffu, v, 4);
      const int o = (lane & 3) * 4 + (h4 ? 2 : 0) + (h3 ? 1 : 0);
      if (!h2)
        *reinterpret_cast<uint32_t*>(smem + F::YST + hu * 256 + (o >> 3) * 128 + (o & 7) * 16 + q * 4) = pack_bf16(v, vi);
    };
    auto smem_mix = [&](uint4 (&wv)[4], int k) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        wv[j] = *reinterpret_cast<const uint4*>(smem + F::MIX + k * 2048 + j * 512 + lane * 16);
    };
    constexpr int kNone = 1 << 20;
    if (F::MIX_ALL) {
      wait(&bar.ldm, par);
#pragma unroll 1
      for (int task = warp; task < F::MIX_TASKS; task += 16) {
        smem_mix(wa, task);
        mix_task(wa, task, kNone);
      }
    } else {
      constexpr int kRest = 32 + F::MIX_TASKS;   // the tasks after those in registers and shared memory
      mix_task(wa, warp, kRest + warp);
      mix_task(wb, warp + 16, kRest + 16 + warp);
      if (warp < F::MIX_TASKS) {
        uint4 wc[4];
        wait(&bar.ldm, par);
        smem_mix(wc, warp);
        mix_task(wc, 32 + warp, kNone);
      }
      mix_task(wa, kRest + warp, kNone);
      if (kRest + 16 + warp < 4 * F::HU) mix_task(wb, kRest + 16 + warp, kNone);
      static_assert(F::MIX_ALL || (kRest + 16 <= 4 * F::HU && 4 * F::HU <= kRest + 32), "tasks");
    }
    proxy_fence();
    tc_before();
    __syncthreads();
    if (warp < CL && lane == 0)
      bulk_s2c(cluster_addr(sm + F::YZ + rank * (F::HU * 256), warp), sm + F::YST, F::HU * 256,
               cluster_addr(smem_addr(&bar.y), warp));
    __syncwarp();
    if (tid == 0) {   // G3 has read X2 and the mode matrices
      if (l + 1 < net.L) {
        mbar_arm(&bar.ldx, 6144);
        bulk_g2s(sm + F::X2, net.dft_x + 4096, 6144, &bar.ldx);
        if (F::MIX_ALL) load_mix_smem(l + 1);
      } else {
        mbar_arm(&bar.ldw, net.H * 64);
        bulk_g2s(sm + F::RECV, net.w1, net.H * 64, &bar.ldw);
      }
    }
    __syncwarp();
    if (warp == 0) {
      // ---- G4
      if (lane == 0) {
        wait1(&bar.lda, par);
        wait1(&bar.y, par);
        mbar_arm(&bar.y, 36864);
        tc_after();
        const PcDesc a(sm + F::YZ, 6144, 128), e(sm + F::EA_EYI, 128, 768);
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
          for (int kk = 0; kk < 3; ++kk)
            pc_mma(tmem + 64 + t * 32, a.at(t * 2048 + kk * 12288), e.at(kk * 256), pc_idesc(2 * ROWS, false), kk > 0);
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
      // K = 24 .. 31: the bias in three parts, exactly, against ones in the inverse x-DFT
      if (tid < ROWS * 32) {
        const float bias = net.pw_b[l * 32 + lane];
        // eight leading bits each, cut off: rounded, the largest finite values would become infinite
        const float hi = fabsf(bias) < INFINITY ? bf_hi(__float_as_uint(bias)) : bias;
        const float mid = hi == bias ? 0.f : bf_hi(__float_as_uint(bias - hi)), lo = hi == bias ? 0.f : (bias - hi) - mid;
        *reinterpret_cast<uint4*>(smem + F::YZ + (tid >> 5) * 2048 + (lane >> 3) * 512 + 384 + (lane & 7) * 16) =
            make_uint4(pack_bf16(hi, mid), pack_bf16(lo, 0.f), 0, 0);
      }
    }
    proxy_fence();
    tc_before();
    __syncthreads();
    // ---- G5: the leader of a set issues its group.  The inverse x-DFT of the group's four rows
    // is one product (N = 4 rows x 32 outputs), the pointwise products follow row by row
    if (leader && set < G) {
      tc_after();
      const uint32_t d = tmem + set * 128;
      const PcDesc x(sm + F::EA, 128, 512), z(sm + F::YZ + set * 8192, 128, 512);
      const PcDesc a(sm + F::ACT + set * 32768, 128, 2048), w(sm + F::EA_PW, 128, 512);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) pc_mma(d, x.at(kk * 256), z.at(kk * 256), pc_idesc(128, false), kk > 0);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
          pc_mma(d + r * 32, a.at(r * 512 + kk * 256), w.at(kk * 256), pc_idesc(32, false), true);
      umma_commit(&bar.g5[set]);
    }
    __syncwarp();
    wait(&bar.g5[grp], par);
    tc_after();
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      uint32_t v[2][16];
      pc_ld<16>(tlane + (grp * 4 + r0 + g) * 32, v[0]);
      pc_ld<16>(tlane + (grp * 4 + r0 + g) * 32 + 16, v[1]);
      pc_ld_wait();
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        uint32_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int o = cc * 8 + 2 * k;
          h[k] = relu_bf16(pack_bf16(__uint_as_float(v[o >> 4][o & 15]), __uint_as_float(v[o >> 4][(o & 15) + 1])));
        }
        *reinterpret_cast<uint4*>(act_px + g * 512 + cc * 128) = make_uint4(h[0], h[1], h[2], h[3]);
      }
    }
    proxy_fence();
    tc_before();
    if (l + 1 < net.L) {
      asm volatile("bar.sync %0, %1;\n" ::"r"(1 + grp), "n"(512 / G) : "memory");   // the group's sets
      if (leader && set < G) {
        tc_after();
        wait1(&bar.ldx, par ^ 1);
        issue_g1(set);
      }
      if (tid == 0) {   // the inverse x-DFT and pointwise operands make way for the y-DFT
        for (int k = 0; k < G; ++k) wait1(&bar.g5[k], par);
        mbar_arm(&bar.ldy, 24576);
        bulk_g2s(sm + F::EA, net.ey, 24576, &bar.ldy);
      }
      __syncwarp();
    }
  }
  __syncthreads();

  // ---- projection, 128 hidden nodes at a time for the four rows of a group: each set takes 32 hidden
  // nodes, whose biases and weights it keeps in registers, and the sets' sums meet in shared
  // memory (with a set per row every bias and weight is a shared-memory or constant-bank read per
  // row: 4200 and 4600 cycles per group, now 3600).
  wait(&bar.ldw, 0);
  float* part = reinterpret_cast<float*>(smem + F::YZ);   // [set][row][128]
  uint32_t ppar = 0;
  const PcDesc pa(sm + F::ACT, 128, 2048), pw(sm + F::RECV, 128, 512);
#pragma unroll 1
  for (int h0 = 0; h0 < net.H; h0 += 128) {
    const int n = min(128, net.H - h0);
    float b1[32], w2[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const int h = set * 32 + k;
      b1[k] = h < n ? net.b1[h0 + h] : 0.f;
      w2[k] = h < n ? net.w2[h0 + h] : 0.f;
    }
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      if (leader) {   // of set: row set of the group
        tc_after();
        const uint32_t idesc = pc_idesc(0, false) | ((uint32_t)(n >> 3) << 17);
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
          pc_mma(tmem + set * 128, pa.at(g * 32768 + set * 512 + kk * 256), pw.at(h0 * 64 + kk * 256), idesc, kk > 0);
        umma_commit(&bar.pr[set]);
      }
      __syncwarp();
#pragma unroll 1
      for (int r = 0; r < 4; ++r) {
        wait(&bar.pr[r], ppar);
        tc_after();
        float acc = 0.f, acc1 = 0.f;
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 16) {
          if (set * 32 + c0 >= n) break;
          uint32_t v[16];
          pc_ld<16>(tlane + r * 128 + set * 32 + c0, v);
          pc_ld_wait();
#pragma unroll
          for (int k = 0; k < 16; k += 2) {
            acc = fmaf(fmaxf(__uint_as_float(v[k]) + b1[c0 + k], 0.f), w2[c0 + k], acc);
            acc1 = fmaf(fmaxf(__uint_as_float(v[k + 1]) + b1[c0 + k + 1], 0.f), w2[c0 + k + 1], acc1);
          }
        }
        part[set * 512 + r * 128 + px] = acc + acc1;
      }
      ppar ^= 1;
      tc_before();
      __syncthreads();
      const int e = set * 128 + px;   // row set of the group, column px
      float* w = wout + ((size_t)b * 128 + y0 + 4 * g + set) * 128 + px;
      const float sum = (part[e] + part[512 + e]) + (part[1024 + e] + part[1536 + e]);
      *w = sum + (h0 == 0 ? net.b2 : *w);
      __syncthreads();
    }
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

// clusters that the current device runs at once (0 if the size cannot be launched), measured once per
// device
template <int CL>
int pc_capacity() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lock(mu);
  const auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  int n = 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  pc_config<CL>(cfg, attr, 1, nullptr);
  if (pc_attributes<CL>() != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, pino_cluster_kernel<CL>, &cfg) != cudaSuccess) {
    cudaGetLastError();   // a size that cannot be launched is not the next call's error
    n = 0;
  }
  cache[dev] = n;
  return n;
}

template <int CL>
int pc_launch(const PinoClusterNet& net, const PinoStates& st, float* wout, int B, int* err, cudaStream_t s) {
  BS_CUDA_TRY(pc_attributes<CL>());
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  pc_config<CL>(cfg, attr, B, s);
  BS_CUDA_TRY(cudaLaunchKernelEx(&cfg, pino_cluster_kernel<CL>, net, st, wout, err));
  return BS_OK;
}

}  // namespace

int launch_pino_cluster(const PinoClusterNet& net, const PinoStates& st, float* wout, int B, int* err,
                        cudaStream_t s) {
  // Clusters of 16 halve every stage's rows (one state 45 us, seven 48, against 62 with 8) while
  // they all run at once; beyond that twice as many clusters of 8 fit (8 states: 62 us, against
  // 96 in two waves of 16; 15 states 65).
  const int c16 = pc_capacity<16>(), c8 = pc_capacity<8>();
  if (c16 > 0 && (c8 == 0 || B <= c16)) return pc_launch<16>(net, st, wout, B, err, s);
  return pc_launch<8>(net, st, wout, B, err, s);
}

}  // namespace bsp
