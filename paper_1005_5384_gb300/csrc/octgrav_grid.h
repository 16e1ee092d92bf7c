// octgrav_grid.h -- cooperative launches: a barrier over the whole grid and the
// launch itself. Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

namespace og {

// Barrier over all blocks of a cooperative launch: every block adds one to
// *bar and waits until it reaches `target` (a multiple of the grid size that
// grows from barrier to barrier). Writes before it are visible to every block
// after it. False when the wait (about 1 s) ran out -- all blocks of a
// cooperative launch are resident, so that would be a lost block; the kernels
// then stop, with `bit` set in *status.
static __device__ bool grid_barrier(int* bar, int target, int* status, int bit) {
  constexpr long long limit = 1ll << 31;  // cycles
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int good = 1, v;
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v - target >= 0) break;  // counts may wrap
      if (clock64() - t0 > limit) {
        atomicOr(status, bit);
        good = 0;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// Blocks of a cooperative launch: at most `most`, and at most eleven twelfths of
// what an idle device holds (the kernel's blocks wait for one another). The device
// starts all of them or none, so a grid that takes every place waits for whatever
// runs on another stream, were it one block that runs for the whole program;
// this one leaves the places of 12 SMs. Five sixths cost 4 % of the levels of a tree
// of a million particles and 24 % of a training step at batch 65,536, eleven
// twelfths 2 and 12 %. 0 on an error.
template <class K>
int resident_blocks(K kernel, int threads, int most, size_t smem = 0) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess)
    return 0;
  return std::min(std::max(1, sms * per * 11 / 12), most);
}

template <class... A>
cudaError_t launch_cooperative(void (*kernel)(A...), int blocks, int threads, size_t smem, cudaStream_t st, A... args) {
  if (blocks < 1) return cudaErrorInvalidConfiguration;
  void* argv[] = {&args...};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kernel), dim3(blocks), dim3(threads), argv, smem, st);
}

}  // namespace og
