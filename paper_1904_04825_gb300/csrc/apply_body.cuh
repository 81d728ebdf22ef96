// Shapes and element types of the element-Jacobi apply, shared by the launches of
// blocks.cu and the GMRES cycle kernel (cycle.cuh).
#pragma once

#include <cuda_bf16.h>

#include "device.cuh"

namespace frk {

template <typename S> struct StoreT;
template <> struct StoreT<double> { __device__ static double to(double x) { return x; } };
template <> struct StoreT<float> { __device__ static float to(float x) { return x; } };
template <> struct StoreT<__nv_bfloat16> {
  __device__ static __nv_bfloat16 to(float x) { return __float2bfloat16_rn(x); }
};
__device__ __forceinline__ double load_acc(const double* p) { return *p; }
__device__ __forceinline__ float load_acc(const float* p) { return *p; }
__device__ __forceinline__ float load_acc(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// z = Minv r (optionally r scaled by *scale first and written back), optional
// sum of squares of z.  EPC elements per CTA, one thread per block row.
// S: block storage type; A: accumulation type (FP64 for FP64 blocks, FP32 otherwise).
// Shape of the staged apply per block size and storage type: KS threads
// share one row's dot product (threads = KS nb), NS elements in flight per
// CTA (element block + its r, one bulk copy each, in a ring of stages).
template <int NB, typename S> struct ApplyShape;
template <> struct ApplyShape<36, double> { static constexpr int KS = 4, NS = 6; };
template <> struct ApplyShape<64, double> { static constexpr int KS = 1, NS = 1; };  // swept: (KS, NS) = (1, 1) 192 us, (1, 2) 197, (2, 2) 201, (2, 3) 218, (4, 3) 231 at 160^2 p=3
template <> struct ApplyShape<100, double> { static constexpr int KS = 2, NS = 2; };
template <> struct ApplyShape<36, float> { static constexpr int KS = 4, NS = 8; };
template <> struct ApplyShape<64, float> { static constexpr int KS = 2, NS = 4; };
template <> struct ApplyShape<100, float> { static constexpr int KS = 2, NS = 3; };
template <> struct ApplyShape<36, __nv_bfloat16> { static constexpr int KS = 4, NS = 8; };
template <> struct ApplyShape<64, __nv_bfloat16> { static constexpr int KS = 2, NS = 6; };
template <> struct ApplyShape<100, __nv_bfloat16> { static constexpr int KS = 2, NS = 4; };
template <> struct ApplyShape<40, double> { static constexpr int KS = 4, NS = 6; };
template <> struct ApplyShape<40, float> { static constexpr int KS = 4, NS = 8; };
template <> struct ApplyShape<40, __nv_bfloat16> { static constexpr int KS = 4, NS = 8; };
template <> struct ApplyShape<144, double> { static constexpr int KS = 1, NS = 1; };
template <> struct ApplyShape<144, float> { static constexpr int KS = 1, NS = 2; };
template <> struct ApplyShape<144, __nv_bfloat16> { static constexpr int KS = 1, NS = 4; };
template <> struct ApplyShape<196, double> { static constexpr int KS = 1, NS = 1; };  // does not fit: rejected
template <> struct ApplyShape<196, float> { static constexpr int KS = 1, NS = 1; };
template <> struct ApplyShape<196, __nv_bfloat16> { static constexpr int KS = 1, NS = 2; };

template <int NB, typename S, typename A>
struct ApplyLayout {
  static constexpr int KS = ApplyShape<NB, S>::KS, NS = ApplyShape<NB, S>::NS;
  static constexpr int WORKERS = KS * NB;                   // threads with a (row, k-range)
  static constexpr int THREADS = (WORKERS + 31) / 32 * 32;  // whole warps (the reductions shuffle)
  static constexpr unsigned MB = (unsigned)(NB * NB * sizeof(S));  // one block (multiple of 16)
  static constexpr unsigned RB = (unsigned)(NB * sizeof(double));  // its r (multiple of 16)
  static constexpr unsigned STAGE = (MB + RB + 127) / 128 * 128;
  static constexpr size_t BYTES = (size_t)NS * STAGE + (size_t)(1 + KS) * NB * sizeof(A) + 32 * sizeof(double) +
                                  NS * sizeof(unsigned long long);
};

// Elements per pass and threads of the one-thread-per-row kernels.
template <int NB> struct RowsShape {
  static constexpr int EPC = NB >= 256 ? 1 : 256 / NB;
  static constexpr int THREADS = (EPC * NB + 31) / 32 * 32;
};

}  // namespace frk
