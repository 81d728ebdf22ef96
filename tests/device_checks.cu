// Device functions of the library called alone, for test_gpu_device_functions.py.
#include <cuda_runtime.h>

#include "cycle.cuh"
#include "gj_fx.cuh"

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

// The common fluxes of n pairs of states, qm and qp [n][4], along direction dir:
// by the operations of R(U) and A z, which give twice the flux, and by those of the
// element blocks.
__global__ void k_fluxes(int n, const double* qm, const double* qp, int kind, int dir, double* fast, double* full) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double a[4];
  frk::riemann_flux2(kind, qm + 4 * i, qp + 4 * i, dir, 1.4, a);
  for (int v = 0; v < 4; ++v) fast[4 * i + v] = 0.5 * a[v];
  frk::riemann_flux(kind, qm + 4 * i, qp + 4 * i, dir, 1.4, a);
  for (int v = 0; v < 4; ++v) full[4 * i + v] = a[v];
}

// rcp_fast and sqrt_fast against the correctly rounded operations at n arguments of
// every exponent that the fast forms take: out[0], out[2] the largest difference in
// units in the last place, out[1], out[3] how many differ.
__global__ void k_rcp_sqrt(unsigned n, unsigned long long* out) {
  const auto bits = [](double x) { return __double_as_longlong(x); };
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    unsigned long long h = (i + 1) * 0x9e3779b97f4a7c15ull;  // a mixed counter: mantissa and exponent
    h = (h ^ (h >> 30)) * 0xbf58476d1ce4e5b9ull;
    h = (h ^ (h >> 27)) * 0x94d049bb133111ebull;
    h ^= h >> 31;
    const unsigned long long e = 0x030 + (h >> 52) % 0x790;
    const double x = __longlong_as_double((long long)(e << 52 | (h & 0xfffffffffffffull)));
    const unsigned long long a = llabs(bits(frk::rcp_fast(x)) - bits(1.0 / x)), b = llabs(bits(frk::sqrt_fast(x)) - bits(sqrt(x)));
    if (a) {
      atomicMax(out, a);
      atomicAdd(out + 1, 1ull);
    }
    if (b) {
      atomicMax(out + 2, b);
      atomicAdd(out + 3, 1ull);
    }
  }
}
// both at given arguments, out [2][n]
__global__ void k_rcp_sqrt_at(int n, const double* x, double* out) {
  const int i = threadIdx.x;
  if (i < n) {
    out[i] = frk::rcp_fast(x[i]);
    out[n + i] = frk::sqrt_fast(x[i]);
  }
}

__global__ void k_max_nonneg(int n, const double* a, const double* b, double* out) {
  if ((int)threadIdx.x < n) out[threadIdx.x] = frk::max_nonneg(a[threadIdx.x], b[threadIdx.x]);
}

// Inverse of the row-major n x n FP64 matrix M, one CTA, by gjfx::invert.
template <int NB> struct InverseLayout {
  static constexpr int LD = NB + 1, THREADS = NB <= 64 ? 128 : 256;
  static constexpr size_t OFF_PIV = (size_t)NB * LD * sizeof(double);
  static constexpr size_t OFF_SCRATCH = (OFF_PIV + NB * sizeof(int) + 127) / 128 * 128;
  static constexpr size_t BYTES = OFF_SCRATCH + frk::gjfx::Shape<NB, THREADS>::BYTES;
};
template <int NB>
__global__ void __launch_bounds__(InverseLayout<NB>::THREADS) k_inverse(const double* M, double* inv) {
  using L = InverseLayout<NB>;
  extern __shared__ __align__(128) unsigned char smem[];
  double* A = reinterpret_cast<double*>(smem);
  int* piv = reinterpret_cast<int*>(smem + L::OFF_PIV);
  unsigned char* scratch = smem + L::OFF_SCRATCH;
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) A[i / NB * L::LD + i % NB] = M[i];
  __syncthreads();
  frk::gjfx::invert<NB, L::LD, L::THREADS>(A, piv, scratch);
  const int* ipr = reinterpret_cast<const int*>(scratch + frk::gjfx::Shape<NB, L::THREADS>::OFF_IPR);
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) inv[i] = A[piv[i / NB] * L::LD + ipr[i % NB]];
}
template <int NB>
int inverse(const double* M, double* inv) {
  using L = InverseLayout<NB>;
  const size_t bytes = sizeof(double) * NB * NB;
  double* dev = nullptr;
  if (cudaMalloc(&dev, 2 * bytes) != cudaSuccess) return -1;
  int rc = -1;
  if (cudaMemcpy(dev, M, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaFuncSetAttribute(k_inverse<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES) == cudaSuccess) {
    k_inverse<NB><<<1, L::THREADS, L::BYTES>>>(dev, dev + NB * NB);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(inv, dev + NB * NB, bytes, cudaMemcpyDeviceToHost) == cudaSuccess)
      rc = 0;
  }
  cudaFree(dev);
  return rc;
}

}  // namespace

// 0 and the inverse of the n x n matrix M (host, row-major), or -1.
extern "C" int fp64_inverse(int n, const double* M, double* inv) {
  switch (n) {
    case 36: return inverse<36>(M, inv);
    case 40: return inverse<40>(M, inv);
    case 64: return inverse<64>(M, inv);
    case 100: return inverse<100>(M, inv);
    case 135: return inverse<135>(M, inv);
    case 144: return inverse<144>(M, inv);
    default: return -1;
  }
}

// 0 and the fluxes (k_fluxes; host arrays), or -1.
extern "C" int fluxes(int n, const double* qm, const double* qp, int kind, int dir, double* fast, double* full) {
  const size_t bytes = (size_t)n * 4 * sizeof(double);
  double* d = nullptr;
  if (n < 1 || cudaMalloc(&d, 4 * bytes) != cudaSuccess) return -1;
  int rc = -1;
  if (cudaMemcpy(d, qm, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaMemcpy(d + 4 * n, qp, bytes, cudaMemcpyHostToDevice) == cudaSuccess) {
    k_fluxes<<<(n + 255) / 256, 256>>>(n, d, d + 4 * n, kind, dir, d + 8 * n, d + 12 * n);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(fast, d + 8 * n, bytes, cudaMemcpyDeviceToHost) == cudaSuccess &&
        cudaMemcpy(full, d + 12 * n, bytes, cudaMemcpyDeviceToHost) == cudaSuccess)
      rc = 0;
  }
  cudaFree(d);
  return rc;
}

extern "C" int rcp_sqrt(unsigned n, unsigned long long* out) {
  unsigned long long* d = nullptr;
  if (cudaMalloc(&d, 4 * sizeof(*out)) != cudaSuccess) return -1;
  int rc = -1;
  if (cudaMemset(d, 0, 4 * sizeof(*out)) == cudaSuccess) {
    k_rcp_sqrt<<<608, 256>>>(n, d);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(out, d, 4 * sizeof(*out), cudaMemcpyDeviceToHost) == cudaSuccess)
      rc = 0;
  }
  cudaFree(d);
  return rc;
}
extern "C" int rcp_sqrt_at(int n, const double* x, double* out) {
  double* d = nullptr;
  if (n < 1 || n > 64 || cudaMalloc(&d, 3 * n * sizeof(double)) != cudaSuccess) return -1;
  int rc = -1;
  if (cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess) {
    k_rcp_sqrt_at<<<1, 64>>>(n, d, d + n);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(out, d + n, 2 * n * sizeof(double), cudaMemcpyDeviceToHost) == cudaSuccess)
      rc = 0;
  }
  cudaFree(d);
  return rc;
}

extern "C" int max_nonneg(int n, const double* a, const double* b, double* out) {
  double* d = nullptr;
  const size_t bytes = n * sizeof(double);
  if (n < 1 || n > 256 || cudaMalloc(&d, 3 * bytes) != cudaSuccess) return -1;
  int rc = -1;
  if (cudaMemcpy(d, a, bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
      cudaMemcpy(d + n, b, bytes, cudaMemcpyHostToDevice) == cudaSuccess) {
    k_max_nonneg<<<1, 256>>>(n, d, d + n, d + 2 * n);
    if (cudaGetLastError() == cudaSuccess && cudaMemcpy(out, d + 2 * n, bytes, cudaMemcpyDeviceToHost) == cudaSuccess) rc = 0;
  }
  cudaFree(d);
  return rc;
}

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
