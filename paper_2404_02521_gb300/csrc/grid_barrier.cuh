// Sums and barriers over the blocks of a cooperative launch (or of a group of its blocks), shared by the
// solvers whose vectors live in global memory.
//
// A barrier is one arrival counter, on which one thread per block waits; the blocks' partial sums
// are read after it.  Measured at 128 blocks, 10.6 us per BiCGSTAB iteration with two of them;
// one slot per block, polled by every block (partial sum and arrival in the same store),
// took the same there and a third longer with 50 or 190 blocks: the polling loads slow each other
// down.  Every wait is bounded: a block that runs out of polls sets bit 1 of the status word,
// which ends the other blocks' waits too, and takes no further part.
#pragma once

#include <cuda_runtime.h>

namespace bsp {

constexpr int kGridPolls = 1 << 22;      // bound on the polls of one barrier
constexpr int kGridMaxBlocks = 1024;     // blocks of a group, as sized in the partial sums

// Whether a counter that only grows has reached the target.  Both are taken modulo 2^32 (a launch of
// 150 blocks passes that in 28 million barriers, minutes of iterations), and a counter is never
// 2^31 away from a target that a block waits for.
__host__ __device__ __forceinline__ bool grid_reached(unsigned seen, unsigned target) {
  return (int)(seen - target) >= 0;
}

struct GridWords {
  float4 partials[2][kGridMaxBlocks];
  unsigned arrivals;   // zero at launch
};

template <int THREADS>
struct GridGroup {
  GridWords* words;     // of this group
  int* status;
  int block, blocks;    // this block's index in the group, blocks of the group
  int tid;
  unsigned target = 0;
  int round = 0;
  bool dead = false;

  __device__ __forceinline__ void barrier() {
    __shared__ int timeout;
    if (dead) return;   // the solve is over: leave without another wait
    target += (unsigned)blocks;
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(&words->arrivals, 1u);
      int polls = 0, out = 0;
      unsigned seen = 0;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(&words->arrivals) : "memory");
        if (grid_reached(seen, target)) break;
        if (++polls >= kGridPolls || ((polls & 1023) == 0 && (*(volatile int*)status & 2))) {
          atomicOr(status, 2);
          out = 1;
          break;
        }
      }
      timeout = out;
    }
    __syncthreads();
    dead = timeout != 0;
  }

  // v summed over the block's threads, bitwise the same in all of them
  __device__ __forceinline__ void block_sum(float (&v)[4]) {
    __shared__ float4 ws[THREADS / 32];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
    if ((tid & 31) == 0) ws[tid >> 5] = make_float4(v[0], v[1], v[2], v[3]);
    __syncthreads();
    v[0] = v[1] = v[2] = v[3] = 0.f;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
      v[0] += ws[w].x; v[1] += ws[w].y; v[2] += ws[w].z; v[3] += ws[w].w;
    }
    __syncthreads();
  }

  // v summed over the group, with a barrier: every block adds the block sums in the same order
  // and returns bitwise the same totals.  The slots alternate, so that a block still reading
  // one round's is not overtaken by the next.
  __device__ __forceinline__ void sum(float (&v)[4]) {
    float4* slot = words->partials[round & 1];
    ++round;
    block_sum(v);
    if (tid == 0) __stcg(slot + block, make_float4(v[0], v[1], v[2], v[3]));
    barrier();
    v[0] = v[1] = v[2] = v[3] = 0.f;
    for (int b = tid; b < blocks; b += THREADS) {
      const float4 q = __ldcg(slot + b);
      v[0] += q.x; v[1] += q.y; v[2] += q.z; v[3] += q.w;
    }
    block_sum(v);
  }
};

}  // namespace bsp
