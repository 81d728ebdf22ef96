// Per-element MLP that predicts a stage solve's initial Krylov guess (not in
// the paper; the GMRES solve still tests the guess and converges to the
// same tolerance).
//
// Network 3nb -> 256 -> 256 -> nb, ReLU, FP32 master weights.
//  * training path (forward with stored activations, backward, Adam): FP32
//    tiled GEMMs on the CUDA cores, so the gradients can be checked against
//    the FP64 oracle;
//  * inference path: BF16 operands on the 5th-generation tensor cores
//    (tcgen05.mma, FP32 accumulator in tensor memory) with bias + ReLU fused
//    into the epilogue that reads the accumulator back.
// Loss: mean of (y - t)^2 / 2 over all outputs; Adam with bias correction.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstring>
#include <new>

#include "device.cuh"
#include "mlp_fused.cuh"

struct fr_mlp {
  int n[4] = {0, 0, 0, 0};  // layer widths: in, hidden, hidden, out
  int max_batch = 0;
  long long nparam = 0;
  float* P = nullptr;       // FP32 master parameters [W1 b1 W2 b2 W3 b3]
  float* G = nullptr;       // gradients (same layout)
  float* Mo = nullptr;      // Adam first moments
  float* Vo = nullptr;      // Adam second moments
  float* Z = nullptr;       // output of the last FP32 forward [M x n[3]]
  float* A[2] = {};         // hidden activations [M x n[l+1]] (positive where the pre-activation is)
  float* D[3] = {};         // loss gradients w.r.t. Z
  float* part = nullptr;    // row splits' partial weight and bias gradients
  __nv_bfloat16* X16 = nullptr;   // BF16 input / hidden activations for inference,
  __nv_bfloat16* H16[2] = {};     //   rows padded to kp[l] (16-byte rows, zero pad)
  __nv_bfloat16* W16[3] = {};     // BF16 weights [n[l+1]][kp[l]], zero-padded columns
  int kp[3] = {0, 0, 0};          // padded widths of the layer inputs
  int* derr = nullptr;            // device flag: a bounded wait of the GEMM gave up
  // TMA tensor maps of the inference operands (input rows, hidden rows, weights)
  // for the weight-stationary GEMM; ws = 1 when every layer's weights fit in
  // shared memory and the maps were built
  CUtensorMap amap[3] = {};       // layer l input: X16 (l = 0), H16[l-1]
  CUtensorMap wmap[3] = {};
  int ws = 0;
  int* herr = nullptr;            // pinned host copy, refreshed after every inference
  double* loss = nullptr;   // device scalar
  int step = 0;
  char err[256] = {0};
};

namespace frk {
namespace {

long long off_W(const fr_mlp* m, int l) {
  long long o = 0;
  for (int i = 0; i < l; ++i) o += (long long)m->n[i + 1] * m->n[i] + m->n[i + 1];
  return o;
}
long long off_b(const fr_mlp* m, int l) { return off_W(m, l) + (long long)m->n[l + 1] * m->n[l]; }

// ---- FP32 tiled GEMM: C(i, j) = sum over k < K of A(i, k) B(k, j) ----
// A is [i][lda] (AK: k runs along memory) or [k][lda]; B is [j][ldb] (BK) or
// [k][ldb].  64 x 64 tile per CTA, 16-deep slices double-buffered in shared
// memory with the next slice's global loads in flight during the FMAs; 128
// threads x (8 x 4) outputs, so a slice step costs 3 16-byte shared loads per 32
// FMAs.  64 x 64 (not 128 x 64) because the batches are 256 to 73,728 rows of 100
// to 300 columns: 8192 rows x 256 columns give 512 CTAs, 3.4 per SM.
// Loads are 16 bytes wide where base, leading dimension and the k range allow
// it (vec), else one value at a time.  One training step of 8192 samples (300-
// 256-256-100), GEMMs and the rest: 5614 -> 412 us; the first version read
// both operands with a stride of one row per lane, summed the bias gradients in
// one thread per column and launched the row splits one after another.
enum SgemmEpilogue {
  EPI_RELU = 0,     // C = max(acc + bias, 0)
  EPI_BIAS2 = 1,    // C = C2 = acc + bias
  EPI_MASK = 2      // C = acc where mask > 0, else 0 (mask laid out as C)
};
struct SgemmArgs {
  int M, N, K;
  const float* A;
  int lda;
  const float* B;
  int ldb;
  float* C;
  int ldc;
  const float* bias;   // EPI_RELU, EPI_BIAS2
  float* C2;           // EPI_BIAS2
  const float* mask;   // EPI_MASK
  int veca, vecb;      // 16-byte loads allowed
};

// four consecutive values along memory at p, `ok` of them in range
__device__ __forceinline__ float4 load4(const float* p, int ok, int vec) {
  if (vec && ok >= 4) return *reinterpret_cast<const float4*>(p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (ok > 0) v.x = p[0];
  if (ok > 1) v.y = p[1];
  if (ok > 2) v.z = p[2];
  if (ok > 3) v.w = p[3];
  return v;
}

constexpr int kGT = 64, kGK = 16, kGP = kGT + 4;  // tile side, slice depth, shared pitch

// this thread's 2 x 4 values of a 64 x 16 operand slice: KC (k along memory):
// row tid / 2, k = 4 (tid % 2) and 8 more (the two halves land 16 banks apart);
// else k = tid / 16 and 8 more, four rows at 4 (tid % 16)
template <bool KC>
__device__ __forceinline__ void slice_load(float4 v[2], const float* X, int ld, int x0, int nx, int k0, int kend,
                                           int vec) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (KC) {
      const int x = x0 + (tid >> 1), k = k0 + 4 * (tid & 1) + 8 * u;
      v[u] = load4(X + (long long)x * ld + k, x < nx ? kend - k : 0, vec);
    } else {
      const int x = x0 + 4 * (tid & 15), k = k0 + (tid >> 4) + 8 * u;
      v[u] = load4(X + (long long)k * ld + x, k < kend ? nx - x : 0, vec);
    }
  }
}
template <bool KC>
__device__ __forceinline__ void slice_store(float (*S)[kGP], const float4 v[2]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (KC) {
      const int x = tid >> 1, k = 4 * (tid & 1) + 8 * u;
      S[k][x] = v[u].x;
      S[k + 1][x] = v[u].y;
      S[k + 2][x] = v[u].z;
      S[k + 3][x] = v[u].w;
    } else {
      *reinterpret_cast<float4*>(&S[(tid >> 4) + 8 * u][4 * (tid & 15)]) = v[u];
    }
  }
}

template <bool AK, bool BK, int EPI>
__global__ void __launch_bounds__(128) k_sgemm(const SgemmArgs a) {
  __shared__ __align__(16) float As[2][kGK][kGP], Bs[2][kGK][kGP];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.y * kGT, j0 = blockIdx.x * kGT;
  const int kend = a.K;
  float acc[8][4] = {};
  float4 va[2], vb[2];
  slice_load<AK>(va, a.A, a.lda, i0, a.M, 0, kend, a.veca);
  slice_load<BK>(vb, a.B, a.ldb, j0, a.N, 0, kend, a.vecb);
  slice_store<AK>(As[0], va);
  slice_store<BK>(Bs[0], vb);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < kend; k0 += kGK) {
    const bool more = k0 + kGK < kend;
    if (more) {
      slice_load<AK>(va, a.A, a.lda, i0, a.M, k0 + kGK, kend, a.veca);
      slice_load<BK>(vb, a.B, a.ldb, j0, a.N, k0 + kGK, kend, a.vecb);
    }
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty + 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][4 * tx]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
    }
    if (more) {  // the other buffer was last read before the previous barrier
      slice_store<AK>(As[buf ^ 1], va);
      slice_store<BK>(Bs[buf ^ 1], vb);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + 8 * ty + u;
    if (i >= a.M) break;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int j = j0 + 4 * tx + v;
      if (j >= a.N) break;
      const long long o = (long long)i * a.ldc + j;
      float c = acc[u][v];
      if (EPI == EPI_RELU) a.C[o] = fmaxf(c + a.bias[j], 0.f);
      if (EPI == EPI_BIAS2) {
        c += a.bias[j];
        a.C[o] = c;
        a.C2[o] = c;
      }
      if (EPI == EPI_MASK) a.C[o] = a.mask[o] > 0.f ? c : 0.f;
    }
  }
}

int vec_ok(const float* p, int ld) { return reinterpret_cast<uintptr_t>(p) % 16 == 0 && ld % 4 == 0; }

template <bool AK, bool BK, int EPI>
void sgemm(SgemmArgs a, cudaStream_t s) {
  a.veca = vec_ok(a.A, a.lda);
  a.vecb = vec_ok(a.B, a.ldb);
  const dim3 grid((a.N + kGT - 1) / kGT, (a.M + kGT - 1) / kGT);
  count_launch();
  k_sgemm<AK, BK, EPI><<<grid, 128, 0, s>>>(a);
}

// ---- weight and bias gradients of all layers in one launch ----
// dW(i, j) = sum over rows r of D(r, i) in(r, j), db(i) = sum of D(r, i), one
// CTA for 32 x 32 outputs of one layer and one part of kPartRows rows: every
// output is one chain of FMAs over its rows in order, because an Adam step
// divides a gradient by its own magnitude and so shows the order of the sums
// wherever a gradient nearly cancels.  The chains leave the outputs as the only
// parallelism, hence the small tile, 2 x 4 outputs a thread (300-256-256-100:
// 176 CTAs a part) and the three layers side by side; D and the layer inputs of
// every layer are kept, so nothing is waited for.  32 rows a stage by cp.async,
// four stages.  A training step of 8192 rows takes 412 us so (5614 with one launch
// per layer and part and strided reads); with 23 shorter chains per output and 64 x
// 64 tiles it took 363, but an element whose gradient nearly cancelled could move
// by 1e-3 of the parameters' size.
constexpr int kPartRows = 4096, kWT = 32, kWStages = 4;
struct WgradArgs {
  int M, first[4];          // rows; first tile of each layer, and their number
  float* out;               // [part][parameters]
  long long stride;
  struct {
    const float *D, *in;    // [M][n], [M][k]
    int n, k, vd, vin;      // widths, 16-byte copies allowed
    long long off;          // weights, biases behind them
  } l[3];
};
// four consecutive floats at x of a row, `ok` of them in range, the rest zero
__device__ __forceinline__ void wgrad_copy4(float* dst, const float* base, long long at, int ok, int vec) {
  const unsigned d = smem_u32(dst);
  if (vec) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(ok >= 4 ? base + at : base),
                 "r"(ok >= 4 ? 16 : 0)
                 : "memory");
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4 * c), "l"(c < ok ? base + at + c : base),
                   "r"(c < ok ? 4 : 0)
                   : "memory");
  }
}
__global__ void __launch_bounds__(128) k_wgrad(const __grid_constant__ WgradArgs a) {
  __shared__ __align__(16) float As[kWStages][kWT][kWT], Bs[kWStages][kWT][kWT];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int tile = blockIdx.x, l = tile >= a.first[2] ? 2 : (tile >= a.first[1] ? 1 : 0);
  const int n = a.l[l].n, k = a.l[l].k, tk = (k + kWT - 1) / kWT;
  const int i0 = (tile - a.first[l]) / tk * kWT, j0 = (tile - a.first[l]) % tk * kWT;
  const int rbeg = blockIdx.y * kPartRows, rend = min(a.M, rbeg + kPartRows), steps = (rend - rbeg + kWT - 1) / kWT;
  const float *D = a.l[l].D, *in = a.l[l].in;
  const int vd = a.l[l].vd, vin = a.l[l].vin;
  const auto load = [&](int step) {
    if (step < steps) {
      const int r0 = rbeg + step * kWT, st = step % kWStages;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int row = (tid >> 3) + 16 * u, c = 4 * (tid & 7), r = r0 + row;
        wgrad_copy4(&As[st][row][c], D, (long long)r * n + i0 + c, r < rend ? n - i0 - c : 0, vd);
        wgrad_copy4(&Bs[st][row][c], in, (long long)r * k + j0 + c, r < rend ? k - j0 - c : 0, vin);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[2][4] = {};
  float asum = 0.f;  // column sum of D, by the first warp of a layer's first column of tiles
#pragma unroll
  for (int st = 0; st < kWStages - 1; ++st) load(st);
  for (int step = 0; step < steps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kWStages - 2) : "memory");
    __syncthreads();  // this stage is filled, and the one before it has been read
    load(step + kWStages - 1);
    const int st = step % kWStages;
#pragma unroll
    for (int kk = 0; kk < kWT; ++kk) {
      const float2 av = *reinterpret_cast<const float2*>(&As[st][kk][2 * ty]);
      const float4 bv = *reinterpret_cast<const float4*>(&Bs[st][kk][4 * tx]);
      acc[0][0] = fmaf(av.x, bv.x, acc[0][0]);
      acc[0][1] = fmaf(av.x, bv.y, acc[0][1]);
      acc[0][2] = fmaf(av.x, bv.z, acc[0][2]);
      acc[0][3] = fmaf(av.x, bv.w, acc[0][3]);
      acc[1][0] = fmaf(av.y, bv.x, acc[1][0]);
      acc[1][1] = fmaf(av.y, bv.y, acc[1][1]);
      acc[1][2] = fmaf(av.y, bv.z, acc[1][2]);
      acc[1][3] = fmaf(av.y, bv.w, acc[1][3]);
    }
    if (j0 == 0 && tid < kWT) {
#pragma unroll
      for (int kk = 0; kk < kWT; ++kk) asum += As[st][kk][tid];
    }
  }
  float* out = a.out + blockIdx.y * a.stride + a.l[l].off;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = i0 + 2 * ty + u, j = j0 + 4 * tx + v;
      if (i < n && j < k) out[(long long)i * k + j] = acc[u][v];
    }
  if (j0 == 0 && tid < kWT && i0 + tid < n) out[(long long)n * k + i0 + tid] = asum;
}

// ---- BF16 tensor-core GEMM for inference: Y = act(X W^T + b) ----
// 5th-generation tensor cores: one thread issues tcgen05.mma (kind::f16,
// BF16 operands, FP32 accumulator in tensor memory), the CTA stages the
// operands in shared memory, and the epilogue reads the accumulator back
// with tcgen05.ld.
//  * CTA tile 128 rows x BN (<= 256) columns, 128 threads (4 warps);
//    K in 64-wide slices through a 2-stage shared-memory ring filled with
//    16-byte cp.async copies (zero-filled outside the matrices), so padded
//    rows/columns contribute exact zeros;
//  * operands K-major without swizzle: 8-row x 16-byte core matrices, the
//    two core matrices of one K=16 step 128 bytes apart (leading byte
//    offset), consecutive 8-row groups 1024 bytes apart (stride byte offset);
//  * one MMA group per slice is committed to that stage's mbarrier; a stage
//    is refilled only after its MMAs completed; every wait is bounded and a
//    wait that gives up sets *err, and the tensor memory is always freed.
// X [M][kp] and W [N][kp] row-major BF16 with kp % 8 == 0 (16-byte rows).
namespace umma {
constexpr int BM = 128, BK = 64, STAGES = 2, MAXN = 256;
constexpr unsigned A_BYTES = BM * BK * 2;        // 16 KB
constexpr unsigned B_BYTES = MAXN * BK * 2;      // 32 KB
constexpr unsigned STAGE_BYTES = A_BYTES + B_BYTES;
constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 64;
constexpr unsigned TMEM_COLS = 256;

// shared-memory matrix descriptor, no swizzle, K-major
__device__ __forceinline__ unsigned long long sdesc(unsigned saddr, unsigned lbo, unsigned sbo) {
  unsigned long long d = 0;
  d |= (unsigned long long)((saddr >> 4) & 0x3FFFu);
  d |= (unsigned long long)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (unsigned long long)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;  // descriptor version (fixed 0b001 at bits 46-48)
  return d;         // base offset 0, absolute-offset mode off, layout 0 = no swizzle
}
// instruction descriptor: FP32 accumulate, BF16 A and B, both K-major, M x N
__host__ __device__ constexpr unsigned idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(m >> 4) << 24);
}
__device__ __forceinline__ void cp16(unsigned dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
}  // namespace umma

template <bool RELU, bool OUT_BF16>
__global__ void __launch_bounds__(128) k_umma_gemm(int M, int N, int kp, const __nv_bfloat16* __restrict__ X,
                                                   const __nv_bfloat16* __restrict__ W,
                                                   const float* __restrict__ bias, void* out, int ldo,
                                                   int* err) {
  using namespace umma;
  extern __shared__ __align__(1024) unsigned char usm[];
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(usm + STAGES * STAGE_BYTES);
  unsigned* tslot = reinterpret_cast<unsigned*>(usm + STAGES * STAGE_BYTES + 32);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * MAXN;
  const int ncol = min(MAXN, N - n0);           // output columns of this tile
  const int bn = (ncol + 15) / 16 * 16;         // MMA N (multiple of 16)
  const int nk = (kp + BK - 1) / BK;
  const unsigned sbase = smem_u32(usm);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < STAGES; ++q) mbar_init(&bar[q], 1);
    mbar_fence_init();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tslot;

  // fill stage st with K slice kt: A rows m0.., B rows n0.. (16-byte chunks)
  auto load = [&](int kt, int st) {
    const unsigned a_s = sbase + st * STAGE_BYTES, b_s = a_s + A_BYTES;
    const int k0 = kt * BK;
    for (int c = tid; c < BM * (BK / 8); c += 128) {
      const int row = c / (BK / 8), kc = c % (BK / 8);
      const int gi = m0 + row, gk = k0 + kc * 8;
      const bool ok = gi < M && gk < kp;
      cp16(a_s + (row / 8) * 1024 + kc * 128 + (row % 8) * 16, ok ? (const void*)(X + (size_t)gi * kp + gk) : (const void*)X, ok);
    }
    for (int c = tid; c < bn * (BK / 8); c += 128) {
      const int row = c / (BK / 8), kc = c % (BK / 8);
      const int gj = n0 + row, gk = k0 + kc * 8;
      const bool ok = gj < N && gk < kp;
      cp16(b_s + (row / 8) * 1024 + kc * 128 + (row % 8) * 16, ok ? (const void*)(W + (size_t)gj * kp + gk) : (const void*)W, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  bool ok = true;
  load(0, 0);
  for (int kt = 0; kt < nk && ok; ++kt) {
    const int st = kt % STAGES;
    if (kt + 1 < nk) {
      const int nst = (kt + 1) % STAGES;
      if (kt + 1 >= STAGES) {  // MMAs of slice kt+1-STAGES must be done with stage nst
        const int u = (kt + 1 - STAGES) / STAGES;
        ok = mbar_wait(&bar[nst], (unsigned)(u & 1), kWaitPolls);
      }
      if (!__syncthreads_and(ok)) break;
      load(kt + 1, nst);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    // generic-proxy writes -> visible to the tensor cores' async proxy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned a_s = sbase + st * STAGE_BYTES, b_s = a_s + A_BYTES;
      const unsigned id = idesc_bf16(BM, bn);
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk) {
        const unsigned long long ad = sdesc(a_s + kk * 256, 128, 1024);
        const unsigned long long bd = sdesc(b_s + kk * 256, 128, 1024);
        const unsigned acc = (kt > 0 || kk > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(id), "r"(acc)
            : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&bar[st]))
                   : "memory");
    }
  }
  // all MMAs done: the last commit tracks every MMA issued before it
  if (ok && nk > 0) {
    const int last = nk - 1;
    ok = mbar_wait(&bar[last % STAGES], (unsigned)((last / STAGES) & 1), kWaitPolls);
  }
  ok = __syncthreads_and(ok);
  if (!ok) {
    asm volatile("cp.async.wait_all;" ::: "memory");  // no copy may land after the CTA leaves
    if (tid == 0) atomicExch(err, 1);
  } else {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // Accumulator -> bias, activation, output type -> a row-major tile of 64
    // rows in the (now idle) stage buffers, then coalesced 16-byte row
    // stores; two passes (warps 0-1, then warps 2-3) keep the staged tile
    // within the stage buffers for FP32 output too.
    using OutT = typename std::conditional<OUT_BF16, __nv_bfloat16, float>::type;
    constexpr int ES = (int)sizeof(OutT);
    const int pitch = bn * ES + 16;  // bytes per staged row (+16 spreads the banks)
    unsigned char* tile = usm;
    const int wcols = min(bn, ldo - n0);  // output columns of this tile
    const bool vec = ((ldo * ES) % 16 == 0) && ((wcols * ES) % 16 == 0);
    for (int pass = 0; pass < 2; ++pass) {
      if ((warp >> 1) == pass) {
        const int lrow = (warp & 1) * 32 + lane;  // row within the pass
        for (int c0 = 0; c0 < bn; c0 += 16) {
          unsigned v[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          float x[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int j = n0 + c0 + q;
            x[q] = __uint_as_float(v[q]) + (j < N ? bias[j] : 0.f);
            if (RELU) x[q] = fmaxf(x[q], 0.f);
          }
          uint4* dst = reinterpret_cast<uint4*>(tile + (size_t)lrow * pitch + (size_t)c0 * ES);
          if (OUT_BF16) {
            unsigned w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * q], x[2 * q + 1]);
              w[q] = *reinterpret_cast<const unsigned*>(&h);
            }
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              dst[q] = make_uint4(__float_as_uint(x[4 * q]), __float_as_uint(x[4 * q + 1]), __float_as_uint(x[4 * q + 2]),
                                  __float_as_uint(x[4 * q + 3]));
          }
        }
      }
      __syncthreads();
      const int r0 = m0 + pass * 64;
      const int rows = max(0, min(64, M - r0));
      if (vec) {
        const int cpr = wcols * ES / 16;  // 16-byte chunks per row
        for (int c = tid; c < rows * cpr; c += 128) {
          const int r = c / cpr, k = c % cpr;
          const uint4 val = *reinterpret_cast<const uint4*>(tile + (size_t)r * pitch + k * 16);
          *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(out) + ((size_t)(r0 + r) * ldo + n0) * ES +
                                    k * 16) = val;
        }
      } else {
        for (int c = tid; c < rows * wcols; c += 128) {
          const int r = c / wcols, k = c % wcols;
          reinterpret_cast<OutT*>(out)[(size_t)(r0 + r) * ldo + n0 + k] =
              reinterpret_cast<const OutT*>(tile + (size_t)r * pitch)[k];
        }
      }
      __syncthreads();
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// x [M][k] FP32 -> y [M][kp] BF16, zero in the padding columns
__global__ void k_f2bf_pad(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, long long M, int k, int kp) {
  const long long n = M * kp;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const long long i = t / kp;
    const int j = (int)(t % kp);
    y[t] = j < k ? __float2bfloat16_rn(x[i * k + j]) : __float2bfloat16_rn(0.f);
  }
}


// dZ_out = (y - t) / (M * n_out), loss partial sums (FP64)
__global__ void k_loss_grad(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ d,
                            long long n, double* loss, Reduce red) {
  __shared__ double sh[32];
  double s = 0.0;
  const float inv = 1.0f / (float)n;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float e = y[i] - t[i];
    d[i] = e * inv;
    s += 0.5 * (double)e * (double)e;
  }
  const double bs = block_sum(s, sh);
  if (threadIdx.x == 0) red.value(0)[blockIdx.x] = bs;
  if (last_block(red.counter)) {
    finish_sums(red, 1, loss);
    if (threadIdx.x == 0) *loss /= (double)n;
  }
}

// sum of the parts' gradients, in order
__global__ void k_sum_parts(const float* __restrict__ part, int nparts, long long n, float* __restrict__ out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int p = 0; p < nparts; ++p) s += part[(long long)p * n + i];
    out[i] = s;
  }
}

// Adam on every parameter, and the BF16 copy of the weights for inference
// (rows padded to kp; the padding stays zero)
struct AdamLayers {
  long long off[3];        // first weight of the layer
  int rows[3], cols[3], kp[3];
  __nv_bfloat16* W16[3];
};
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                       float c1, float c2, const AdamLayers al) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float x = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = x;
    const int l = i >= al.off[2] ? 2 : (i >= al.off[1] ? 1 : 0);
    const long long w = i - al.off[l];
    if (w < (long long)al.rows[l] * al.cols[l]) {
      const int r = (int)(w / al.cols[l]), c = (int)(w % al.cols[l]);
      al.W16[l][(long long)r * al.kp[l] + c] = __float2bfloat16_rn(x);
    }
  }
}

int mlp_err(fr_mlp* m, int code, const char* msg) {
  if (m) {
    std::strncpy(m->err, msg, sizeof(m->err) - 1);
    m->err[sizeof(m->err) - 1] = 0;
  }
  return code;
}

#define MLP_CUDA(m, call)                                                  \
  do {                                                                     \
    cudaError_t e_ = (call);                                               \
    if (e_ != cudaSuccess) return mlp_err((m), FR_ERR_CUDA, cudaGetErrorString(e_)); \
  } while (0)

unsigned grid_for(long long n) {
  long long g = (n + 255) / 256;
  if (g > 4096) g = 4096;
  return (unsigned)(g < 1 ? 1 : g);
}

// BF16 copies of the weights with rows padded to 16 bytes (biases stay FP32)
int refresh_bf16(fr_mlp* m, cudaStream_t s) {
  for (int l = 0; l < 3; ++l) {
    const long long n = (long long)m->n[l + 1] * m->kp[l];
    count_launch();
    k_f2bf_pad<<<grid_for(n), 256, 0, s>>>(m->P + off_W(m, l), m->W16[l], m->n[l + 1], m->n[l], m->kp[l]);
  }
  MLP_CUDA(m, cudaGetLastError());
  return FR_OK;
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 2D BF16 row-major [rows][ld] (cols <= ld valid), boxes of 64 columns x box_rows
// rows, 128-byte swizzle, zero fill outside
bool make_map(CUtensorMap* map, const void* base, long long rows, int cols, int ld, int box_rows) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)umws::BK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// tensor maps of the weight-stationary inference (all three layers, or none)
void build_maps(fr_mlp* m) {
  m->ws = 0;
  for (int l = 0; l < 3; ++l)
    if (!umws::fits(m->n[l + 1], m->kp[l])) return;
  for (int l = 0; l < 3; ++l) {
    const void* in = l == 0 ? (const void*)m->X16 : (const void*)m->H16[l - 1];
    if (!make_map(&m->amap[l], in, m->max_batch, m->kp[l], m->kp[l], umws::BM)) return;
    if (!make_map(&m->wmap[l], m->W16[l], m->n[l + 1], m->kp[l], m->kp[l], umws::npad_of(m->n[l + 1]))) return;
  }
  m->ws = 1;
}

void free_mlp(fr_mlp* m) {
  if (!m) return;
  cudaFree(m->P); cudaFree(m->G); cudaFree(m->Mo); cudaFree(m->Vo);
  for (auto* p : m->W16) cudaFree(p);
  cudaFree(m->derr);
  cudaFreeHost(m->herr);
  cudaFree(m->Z);
  for (auto* p : m->A) cudaFree(p);
  for (auto* p : m->D) cudaFree(p);
  cudaFree(m->part); cudaFree(m->X16);
  for (auto* p : m->H16) cudaFree(p);
  cudaFree(m->loss);
  delete m;
}

// Reduction scratch for the loss (own copy, independent of any fr_ctx).
struct MlpRed {
  double* partials = nullptr;
  unsigned* counter = nullptr;
};
MlpRed g_mlp_red[64];

}  // namespace
}  // namespace frk

using namespace frk;

extern "C" int fr_mlp_create(int n_in, int n_hidden, int n_out, int max_batch, fr_mlp** out) {
  if (!out) return FR_ERR_INVALID_ARG;
  *out = nullptr;
  if (n_in < 1 || n_hidden < 1 || n_out < 1 || max_batch < 1) return FR_ERR_INVALID_ARG;
  fr_mlp* m = new (std::nothrow) fr_mlp();
  if (!m) return FR_ERR_CUDA;
  m->n[0] = n_in; m->n[1] = n_hidden; m->n[2] = n_hidden; m->n[3] = n_out;
  m->max_batch = max_batch;
  m->nparam = off_b(m, 2) + n_out;
  auto fail = [&](cudaError_t e) { free_mlp(m); return e == cudaSuccess ? FR_OK : FR_ERR_CUDA; };
  cudaError_t e = cudaSuccess;
  const size_t np = (size_t)m->nparam;
  if (e == cudaSuccess) e = cudaMalloc(&m->P, np * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&m->G, np * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&m->Mo, np * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&m->Vo, np * sizeof(float));
  for (int l = 0; l < 3; ++l) m->kp[l] = (m->n[l] + 7) / 8 * 8;
  for (int l = 0; l < 3 && e == cudaSuccess; ++l)
  {
    const size_t wb = (size_t)m->n[l + 1] * m->kp[l] * sizeof(__nv_bfloat16);
    e = cudaMalloc(&m->W16[l], wb);
    if (e == cudaSuccess) e = cudaMemset(m->W16[l], 0, wb);
  }
  if (e == cudaSuccess) e = cudaMalloc(&m->derr, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(m->derr, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMallocHost(&m->herr, sizeof(int));
  if (e == cudaSuccess) *m->herr = 0;
  if (e == cudaSuccess) e = cudaMalloc(&m->Z, (size_t)max_batch * n_out * sizeof(float));
  for (int l = 0; l < 3 && e == cudaSuccess; ++l)
    e = cudaMalloc(&m->D[l], (size_t)max_batch * m->n[l + 1] * sizeof(float));
  for (int l = 0; l < 2 && e == cudaSuccess; ++l) {
    e = cudaMalloc(&m->A[l], (size_t)max_batch * m->n[l + 1] * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&m->H16[l], (size_t)max_batch * m->kp[l + 1] * sizeof(__nv_bfloat16));
  }
  const int parts = (max_batch + kPartRows - 1) / kPartRows;
  if (e == cudaSuccess && parts > 1) e = cudaMalloc(&m->part, (size_t)parts * np * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&m->X16, (size_t)max_batch * m->kp[0] * sizeof(__nv_bfloat16));
  if (e == cudaSuccess) e = cudaMalloc(&m->loss, sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(m->Mo, 0, np * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(m->Vo, 0, np * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(m->P, 0, np * sizeof(float));
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess && dev >= 0 && dev < 64 && !g_mlp_red[dev].partials) {
    e = cudaMalloc(&g_mlp_red[dev].partials, (size_t)kRedBlocks * kMaxVec * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&g_mlp_red[dev].counter, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(g_mlp_red[dev].counter, 0, sizeof(unsigned));
  }
  if (e != cudaSuccess) return fail(e);
  build_maps(m);
  *out = m;
  return FR_OK;
}

extern "C" int fr_mlp_destroy(fr_mlp* m) {
  free_mlp(m);
  return FR_OK;
}

extern "C" const char* fr_mlp_last_error(const fr_mlp* m) { return m ? m->err : "invalid model"; }

extern "C" long long fr_mlp_num_params(const fr_mlp* m) { return m ? m->nparam : 0; }

extern "C" int fr_mlp_set_params(fr_mlp* m, const float* host, void* stream) {
  if (!m || !host) return FR_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  MLP_CUDA(m, cudaMemcpyAsync(m->P, host, m->nparam * sizeof(float), cudaMemcpyHostToDevice, s));
  MLP_CUDA(m, cudaMemsetAsync(m->Mo, 0, m->nparam * sizeof(float), s));
  MLP_CUDA(m, cudaMemsetAsync(m->Vo, 0, m->nparam * sizeof(float), s));
  m->step = 0;
  FRK_TRY(refresh_bf16(m, s));
  MLP_CUDA(m, cudaStreamSynchronize(s));
  return FR_OK;
}

extern "C" int fr_mlp_get_params(fr_mlp* m, float* host, void* stream) {
  if (!m || !host) return FR_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  MLP_CUDA(m, cudaMemcpyAsync(host, m->P, m->nparam * sizeof(float), cudaMemcpyDeviceToHost, s));
  MLP_CUDA(m, cudaStreamSynchronize(s));
  return FR_OK;
}

extern "C" int fr_mlp_get_grads(fr_mlp* m, float* host, void* stream) {
  if (!m || !host) return FR_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  MLP_CUDA(m, cudaMemcpyAsync(host, m->G, m->nparam * sizeof(float), cudaMemcpyDeviceToHost, s));
  MLP_CUDA(m, cudaStreamSynchronize(s));
  return FR_OK;
}

extern "C" int fr_mlp_forward(fr_mlp* m, const float* X, int M, float* Y, int bf16, void* stream) {
  if (!m || !X || !Y || M < 1 || M > m->max_batch) return mlp_err(m, FR_ERR_INVALID_ARG, "bad forward arguments");
  if (*m->herr) return mlp_err(m, FR_ERR_TIMEOUT, "an earlier tensor-core GEMM gave up a bounded wait");
  cudaStream_t s = as_stream(stream);
  if (!bf16) {
    const float* in = X;
    for (int l = 0; l < 3; ++l) {
      SgemmArgs g{};
      g.M = M; g.N = m->n[l + 1]; g.K = m->n[l];
      g.A = in; g.lda = m->n[l];
      g.B = m->P + off_W(m, l); g.ldb = m->n[l];
      g.bias = m->P + off_b(m, l);
      g.C = l < 2 ? m->A[l] : Y; g.ldc = g.N;
      g.C2 = m->Z;
      if (l < 2) sgemm<true, true, EPI_RELU>(g, s);
      else sgemm<true, true, EPI_BIAS2>(g, s);
      in = g.C;
    }
  } else {
    static bool attr = false;  // dynamic shared memory above 48 KB, set once per process
    if (!attr) {
      MLP_CUDA(m, cudaFuncSetAttribute(k_umma_gemm<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)umma::SMEM));
      MLP_CUDA(m, cudaFuncSetAttribute(k_umma_gemm<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)umma::SMEM));
      attr = true;
    }
    // the whole network in one kernel where the call's widths and rows allow it (mlp_fused.cuh)
    if (m->ws && mlpf::takes(m->n, X, Y, M)) {
      MLP_CUDA(m, cudaFuncSetAttribute(mlpf::k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mlpf::BYTES));
      int sms = 0, dev = 0;
      MLP_CUDA(m, cudaGetDevice(&dev));
      MLP_CUDA(m, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      mlpf::Layers L;
      for (int l = 0; l < 4; ++l) L.n[l] = m->n[l];
      for (int l = 0; l < 3; ++l) {
        L.kp[l] = m->kp[l];
        L.bias[l] = m->P + off_b(m, l);
      }
      const int tiles = (M + umws::BM - 1) / umws::BM;
      count_launch();
      mlpf::k_mlp_fused<<<std::min(tiles, sms), mlpf::THREADS, mlpf::BYTES, s>>>(m->wmap[0], m->wmap[1], m->wmap[2], L, X, M,
                                                                               Y, m->derr);
      MLP_CUDA(m, cudaGetLastError());
      MLP_CUDA(m, cudaMemcpyAsync(m->herr, m->derr, sizeof(int), cudaMemcpyDeviceToHost, s));
      return FR_OK;
    }
    count_launch();
    k_f2bf_pad<<<grid_for((long long)M * m->kp[0]), 256, 0, s>>>(X, m->X16, M, m->n[0], m->kp[0]);
    if (m->ws) {
      // weight-stationary persistent GEMMs: one CTA per SM (at most one per 128-row tile)
      static int sms = 0;
      if (sms == 0) {
        int dev = 0;
        MLP_CUDA(m, cudaGetDevice(&dev));
        MLP_CUDA(m, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        MLP_CUDA(m, cudaFuncSetAttribute(umws::k_umma_ws<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)umws::kSmemLimit));
        MLP_CUDA(m, cudaFuncSetAttribute(umws::k_umma_ws<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)umws::kSmemLimit));
      }
      const int tiles = (M + umws::BM - 1) / umws::BM;
      const unsigned grid = (unsigned)std::min(tiles, sms);
      for (int l = 0; l < 3; ++l) {
        const int N = m->n[l + 1];
        const size_t smem = umws::smem_bytes(N, m->kp[l]);
        count_launch();
        if (l < 2)
          umws::k_umma_ws<true, true><<<grid, umws::THREADS, smem, s>>>(m->amap[l], m->wmap[l], M, N, m->kp[l],
                                                                        m->P + off_b(m, l), m->H16[l], m->kp[l + 1],
                                                                        m->derr);
        else
          umws::k_umma_ws<false, false><<<grid, umws::THREADS, smem, s>>>(m->amap[l], m->wmap[l], M, N, m->kp[l],
                                                                          m->P + off_b(m, l), Y, N, m->derr);
      }
      MLP_CUDA(m, cudaGetLastError());
      MLP_CUDA(m, cudaMemcpyAsync(m->herr, m->derr, sizeof(int), cudaMemcpyDeviceToHost, s));
      return FR_OK;
    }
    const __nv_bfloat16* in = m->X16;
    for (int l = 0; l < 3; ++l) {
      const int N = m->n[l + 1];
      const dim3 grid((M + umma::BM - 1) / umma::BM, (N + umma::MAXN - 1) / umma::MAXN);
      count_launch();
      if (l < 2)
        k_umma_gemm<true, true><<<grid, 128, umma::SMEM, s>>>(M, N, m->kp[l], in, m->W16[l], m->P + off_b(m, l),
                                                              m->H16[l], m->kp[l + 1], m->derr);
      else
        k_umma_gemm<false, false><<<grid, 128, umma::SMEM, s>>>(M, N, m->kp[l], in, m->W16[l], m->P + off_b(m, l),
                                                                Y, N, m->derr);
      in = l < 2 ? m->H16[l] : nullptr;
    }
  }
  MLP_CUDA(m, cudaGetLastError());
  // the GEMMs' error flag reaches the host with the stream; the next call reports it
  if (bf16) MLP_CUDA(m, cudaMemcpyAsync(m->herr, m->derr, sizeof(int), cudaMemcpyDeviceToHost, s));
  return FR_OK;
}

extern "C" int fr_mlp_backward(fr_mlp* m, const float* X, const float* T, int M, double* loss_host,
                               void* stream) {
  if (!m || !X || !T || M < 1 || M > m->max_batch) return mlp_err(m, FR_ERR_INVALID_ARG, "bad backward arguments");
  cudaStream_t s = as_stream(stream);
  int dev = 0;
  MLP_CUDA(m, cudaGetDevice(&dev));
  Reduce red{g_mlp_red[dev].partials, g_mlp_red[dev].counter};
  const long long nout = (long long)M * m->n[3];
  // Z holds the forward pass's output
  count_launch();
  k_loss_grad<<<grid_for(nout) > 1024 ? 1024 : grid_for(nout), 256, 0, s>>>(m->Z, T, m->D[2], nout, m->loss, red);
  for (int l = 2; l > 0; --l) {  // D[l-1] = D[l] W_l where the activation is positive
    SgemmArgs d{};
    d.M = M; d.N = m->n[l]; d.K = m->n[l + 1];
    d.A = m->D[l]; d.lda = d.K;
    d.B = m->P + off_W(m, l); d.ldb = d.N;
    d.C = m->D[l - 1]; d.ldc = d.N;
    d.mask = m->A[l - 1];
    sgemm<true, false, EPI_MASK>(d, s);
  }
  const int parts = (M + kPartRows - 1) / kPartRows;
  WgradArgs g{};
  g.M = M;
  g.out = parts > 1 ? m->part : m->G;
  g.stride = m->nparam;
  for (int l = 0; l < 3; ++l) {
    const int n = m->n[l + 1], k = m->n[l];
    g.l[l].D = m->D[l];
    g.l[l].in = l == 0 ? X : m->A[l - 1];
    g.l[l].n = n;
    g.l[l].k = k;
    g.l[l].vd = vec_ok(g.l[l].D, n);
    g.l[l].vin = vec_ok(g.l[l].in, k);
    g.l[l].off = off_W(m, l);
    g.first[l + 1] = g.first[l] + ((n + kWT - 1) / kWT) * ((k + kWT - 1) / kWT);
  }
  count_launch();
  k_wgrad<<<dim3(g.first[3], parts), 128, 0, s>>>(g);
  if (parts > 1) {
    count_launch();
    k_sum_parts<<<grid_for(m->nparam), 256, 0, s>>>(m->part, parts, m->nparam, m->G);
  }
  MLP_CUDA(m, cudaGetLastError());
  if (loss_host) {
    MLP_CUDA(m, cudaMemcpyAsync(loss_host, m->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    MLP_CUDA(m, cudaStreamSynchronize(s));
  }
  return FR_OK;
}

extern "C" int fr_mlp_adam(fr_mlp* m, float lr, float beta1, float beta2, float eps, void* stream) {
  if (!m) return FR_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  m->step += 1;
  const float c1 = 1.f - std::pow(beta1, (float)m->step);
  const float c2 = 1.f - std::pow(beta2, (float)m->step);
  AdamLayers al;
  for (int l = 0; l < 3; ++l) {
    al.off[l] = off_W(m, l);
    al.rows[l] = m->n[l + 1];
    al.cols[l] = m->n[l];
    al.kp[l] = m->kp[l];
    al.W16[l] = m->W16[l];
  }
  count_launch();
  k_adam<<<grid_for(m->nparam), 256, 0, s>>>(m->P, m->G, m->Mo, m->Vo, m->nparam, lr, beta1, beta2, eps, c1, c2, al);
  MLP_CUDA(m, cudaGetLastError());
  return FR_OK;
}
