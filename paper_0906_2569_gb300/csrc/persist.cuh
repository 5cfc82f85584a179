// Grid barrier and work queue of the persistent batched H|psi> kernels.  Every wait is bounded: on expiry the CTA
// raises the context's error word and leaves.  Included inside an anonymous namespace of namespace hpsi.
#pragma once

constexpr long long kPersistWait = 2000000000LL;   // clock cycles (about 1 s) per barrier wait

__device__ __forceinline__ bool persist_sync(unsigned* bar, unsigned target, int* err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    int good = 1;
    const long long t0 = clock64();
    for (unsigned spins = 0;; ++spins) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((spins & 255u) == 255u && (*(volatile int*)err != 0 || clock64() - t0 > kPersistWait)) {
        atomicCAS(err, 0, 3);
        good = 0;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// The CTA's next tile of a phase (all threads get the same index).
__device__ __forceinline__ int persist_next(unsigned* ctr) {
  __shared__ int tile;
  __syncthreads();   // the previous tile is done with shared memory and with `tile`
  if (threadIdx.x == 0) tile = (int)atomicAdd(ctr, 1u);
  __syncthreads();
  return tile;
}
