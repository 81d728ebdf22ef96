// Device functions of the library called alone, for test_gpu_device_functions.py.
#include <cuda_runtime.h>

#include "cycle.cuh"

namespace {

// Rounds of the grid barrier from a given counter: every CTA notes the round before
// a barrier and checks the others' notes behind it; the last CTA sets the done bit
// with every third round and clears it with the next.
__global__ void k_barrier_rounds(unsigned* counter, unsigned start, int* notes, int rounds, int* errors) {
  __shared__ frk::cyc::Shared s;
  frk::cyc::Grid g{counter, start, 1u << 22, (int)blockIdx.x, (int)gridDim.x, true};
  const bool keeper = g.bid == g.nblk - 1;
  for (int r = 0; r < rounds; ++r) {
    if (threadIdx.x == 0) *(volatile int*)(notes + g.bid) = r;
    const unsigned add = r % 3 == 0 ? frk::cyc::kDone : (r % 3 == 1 ? 0u - frk::cyc::kDone : 0u);
    if (!frk::cyc::barrier(g, s, keeper ? add : 0u)) {
      if (threadIdx.x == 0) atomicAdd(errors, 1);
      return;
    }
    if (threadIdx.x < g.nblk && *(volatile int*)(notes + threadIdx.x) < r) atomicAdd(errors, 1);
    if (threadIdx.x == 0 && s.flag != (r % 3 == 0)) atomicAdd(errors, 1);
    if (!frk::cyc::barrier(g, s)) {  // all have looked before the next note
      if (threadIdx.x == 0) atomicAdd(errors, 1);
      return;
    }
  }
}

}  // namespace

// Errors of `rounds` rounds over nblk CTAs from the counter value `start`, or -1.
extern "C" int check_barrier(int nblk, unsigned start, int rounds) {
  unsigned* dev = nullptr;
  if (nblk < 1 || nblk > 32 || cudaMalloc(&dev, (2 + nblk) * sizeof(int)) != cudaSuccess) return -1;
  int out = -1;
  int* errors = reinterpret_cast<int*>(dev + 1);
  int* notes = errors + 1;
  void* args[] = {&dev, &start, &notes, &rounds, &errors};
  if (cudaMemset(dev, 0, (2 + nblk) * sizeof(int)) == cudaSuccess &&
      cudaMemcpy(dev, &start, sizeof(start), cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaLaunchCooperativeKernel((const void*)k_barrier_rounds, dim3(nblk), dim3(64), args, 0, 0) == cudaSuccess &&
      cudaDeviceSynchronize() == cudaSuccess) {
    int got = 0;
    if (cudaMemcpy(&got, errors, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess) out = got;
  }
  cudaFree(dev);
  return out;
}
