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
constexpr int kGridMaxBlocks = 1024;     // blocks of a launch

// Whether a counter that only grows has reached the target.  Both are taken modulo 2^32 (a launch of
// 150 blocks passes that in 28 million barriers, minutes of iterations), and a counter is never
// 2^31 away from a target that a block waits for.
__host__ __device__ __forceinline__ bool grid_reached(unsigned seen, unsigned target) {
  return (int)(seen - target) >= 0;
}

template <int THREADS>
struct GridGroup {
  unsigned* arrivals;   // of this group, zero at launch
  float4* partials;     // [2][stride] sums of the group's tiles or blocks
  int stride;
  int* status;
  int block, blocks;    // this block's index in the group, blocks of the group
  int tid;
  unsigned target = 0;
  int round = 0;
  bool dead = false;
  int pending = -1;     // slot whose sums wait in shared memory, and the half that they wait in
  int half = 0;

  __device__ __forceinline__ void barrier() {
    __shared__ int timeout;
    if (dead) return;   // the solve is over: leave without another wait
    target += (unsigned)blocks;
    __syncthreads();
    flush();
    if (tid == 0) {
      // releases what the block wrote before its own barrier
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(arrivals) : "memory");
      int polls = 0, out = 0;
      unsigned seen = 0;
      while (true) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(arrivals) : "memory");
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

  // v summed over the block's threads, bitwise the same in all of them.  Its calls lie block barriers
  // apart, so a warp may still read the sums when the others go on.
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
  }

  // The group's sum of v in two halves: a slot takes the block's sum for one of its tiles, and the
  // total of `count` slots follows behind a barrier.  Every block adds the slots in the same order
  // and returns bitwise the same totals, which depend on the tiles and not on the blocks that
  // own them.  The slots alternate, so that a block still reading one round's is not overtaken by
  // the next.
  // put() needs no barrier of its own: the warps' sums wait in one of two shared arrays until flush(),
  // which follows the next block barrier.
  __device__ __forceinline__ static float4* waiting() {
    __shared__ float4 ws[2 * (THREADS / 32)];
    return ws;
  }
  __device__ __forceinline__ void put(float (&v)[4], int slot) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
    if ((tid & 31) == 0) waiting()[half * (THREADS / 32) + (tid >> 5)] = make_float4(v[0], v[1], v[2], v[3]);
    pending = slot;
  }
  __device__ __forceinline__ void flush() {
    if (pending < 0) return;
    if (tid == 0) {
      const float4* ws = waiting() + half * (THREADS / 32);
      float4 s = ws[0];
#pragma unroll
      for (int w = 1; w < THREADS / 32; ++w) {
        s.x += ws[w].x; s.y += ws[w].y; s.z += ws[w].z; s.w += ws[w].w;
      }
      __stcg(partials + (round & 1) * stride + pending, s);
    }
    pending = -1;
    half ^= 1;
  }
  __device__ __forceinline__ void total(float (&v)[4], int count) {
    barrier();
    const float4* slot = partials + (round & 1) * stride;
    ++round;
    v[0] = v[1] = v[2] = v[3] = 0.f;
    // (every warp adding all the slots by itself needs no block barrier and is slower by up to half: the
    // blocks' loads of the same lines queue)
    for (int b = tid; b < count; b += THREADS) {
      const float4 q = __ldcg(slot + b);
      v[0] += q.x; v[1] += q.y; v[2] += q.z; v[3] += q.w;
    }
    block_sum(v);
  }
  __device__ __forceinline__ void sum(float (&v)[4]) {   // with a slot per block
    put(v, block);
    total(v, blocks);
  }
};

}  // namespace bsp
