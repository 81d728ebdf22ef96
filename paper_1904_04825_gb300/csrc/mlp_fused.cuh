// The guess network's whole BF16 inference in one kernel: Y = W3 relu(W2 relu(W1 x
// + b1) + b2) + b3 for 128-row tiles of X, hidden activations in tensor memory.
//
// Layer by layer (umma_ws.cuh) the activations cross memory three times as BF16
// after a conversion pass; here X is read once in FP32 and Y written once, and
// the weights (345 KB at 300-256-256-100, more than an SM holds) stream from L2
// by TMA in slices of 64 columns.  Persistent CTAs, one per SM, tile =
// blockIdx.x + i gridDim.x:
//  * warp 0 streams the slices of W1, W2, W3, tile after tile, through four stages;
//  * warp 1 issues the MMAs (tcgen05.mma kind::f16, FP32 accumulators in tensor
//    memory), slice by slice and K step by K step in the order of the layer
//    kernels, so the results are the same bits;
//  * warps 2..17 take each layer's accumulator, add the bias, apply ReLU, and
//    write the next layer's operand back to tensor memory as BF16 (the MMAs of
//    layers 2 and 3 read A there: no pass through shared memory, whose room goes
//    to the weight stages), or store Y;
//  * warps 18..25 read the next tile's rows of X, round them to BF16 and write the
//    128-byte-swizzled operand as soon as layer 1 has read the tile before.
// Tensor memory: columns 0..255 the hidden layers' accumulator, 256..383 H,
// 384..511 the output's, so layer 1 of the next tile runs beside this tile's
// output.  The layers of one tile follow one another, each with an epilogue of
// 1-2.5 us, and this chain (about 10 us a tile) bounds the kernel, not the MMAs
// (3 us), the weights or X.
// 73,728 rows of 300-256-256-100: 51 us, 157 us as four kernels; X and Y alone
// take 17 us at the HBM rate.
// Every wait is bounded; a wait that gives up sets *err, and copies and MMAs that
// were issued are waited for (bounded) before the tensor memory is freed.
#pragma once

#include "umma_ws.cuh"

namespace frk {
namespace mlpf {

using umws::BK;
using umws::BM;
constexpr int WSTAGES = 4, EPI_WARPS = 16, LOAD_WARPS = 8, THREADS = 32 * (2 + EPI_WARPS + LOAD_WARPS);
constexpr unsigned SLICE = BM * BK * 2;       // an operand slice: 128 rows x 64 columns
constexpr unsigned WSTAGE = 256 * BK * 2;     // a weight slice of up to 256 rows
constexpr int XK = 5;                         // slices of X: inputs up to 320 wide
constexpr int MAX_HIDDEN = 256, MAX_OUT = 128;
constexpr unsigned COL_H = 256, COL_OUT = 384;  // tensor memory: hidden accumulator, H (two BF16 a column), output accumulator
constexpr size_t OFF_W = (size_t)XK * SLICE, OFF_BIAS = OFF_W + (size_t)WSTAGES * WSTAGE,
                 OFF_BAR = OFF_BIAS + 3 * 256 * 4, BYTES = OFF_BAR + 24 * 8 + 1024;  // + alignment slack
static_assert(BYTES <= umws::kSmemLimit, "shared memory");

// The calls this kernel takes: widths that its buffers hold, rows of X and Y that 16-byte
// accesses can take, and no overlap of X and Y (tiles of Y are written while other tiles
// of X are still to be read).
inline bool takes(const int n[4], const float* X, const float* Y, long long M) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(X), y = reinterpret_cast<uintptr_t>(Y);
  return n[0] <= XK * BK && n[0] % 4 == 0 && n[1] <= MAX_HIDDEN && n[2] <= MAX_HIDDEN && n[3] <= MAX_OUT && x % 16 == 0 && y % 16 == 0 &&
         (x + 4ull * M * n[0] <= y || y + 4ull * M * n[3] <= x);
}

struct Layers {
  int n[4];                // widths
  int kp[3];               // padded input widths
  const float* bias[3];
};

__device__ __forceinline__ void commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// a wait of a whole warp, with one answer
__device__ __forceinline__ bool warp_wait(unsigned long long* bar, unsigned parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, kWaitPolls));
}
// 16 accumulator columns of this thread's row
__device__ __forceinline__ void tmem_ld16(unsigned (&v)[16], unsigned addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(addr));
}
// two FP32 sums, each rounded as one
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
// 4 x 4 transposition over four neighbouring lanes of the 16-byte pieces (x[2k], x[2k + 1])
__device__ __forceinline__ void transpose4(float2 (&x)[8], int lane) {
#pragma unroll
  for (int d = 1; d <= 2; d *= 2) {
    const bool up = lane & d;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k & d) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float2 &lo = x[2 * k + h], &hi = x[2 * (k + d) + h];
        const float sx = __shfl_xor_sync(0xffffffffu, up ? lo.x : hi.x, d);
        const float sy = __shfl_xor_sync(0xffffffffu, up ? lo.y : hi.y, d);
        if (up) lo = make_float2(sx, sy);
        else hi = make_float2(sx, sy);
      }
    }
  }
}
// 16-byte chunk of column c (a multiple of 8) in row r of an operand
__device__ __forceinline__ unsigned chunk_of(int r, int c) {
  return (unsigned)(c >> 6) * SLICE + (unsigned)r * 128u + (unsigned)((((c & 63) >> 3) ^ (r & 7)) << 4);
}

__global__ void __launch_bounds__(THREADS, 1)
    k_mlp_fused(const __grid_constant__ CUtensorMap w1, const __grid_constant__ CUtensorMap w2,
                const __grid_constant__ CUtensorMap w3, const __grid_constant__ Layers L, const float* __restrict__ X, int M,
                float* __restrict__ Y, int* err) {
  extern __shared__ unsigned char raw[];
  unsigned char* sm =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* Xs = sm;
  unsigned char* Ws = sm + OFF_W;
  float* bias_s = reinterpret_cast<float*>(sm + OFF_BIAS);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(sm + OFF_BAR);
  unsigned long long *xfull = bar, *xfree = bar + 1, *hfull = bar + 2 /* 2 */, *tfull = bar + 4 /* 3 */,
                     *wfull = bar + 7 /* WSTAGES */, *wempty = wfull + WSTAGES;
  unsigned* tslot = reinterpret_cast<unsigned*>(wempty + WSTAGES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = (M + BM - 1) / BM;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(umws::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    mbar_init(xfull, LOAD_WARPS);
    mbar_init(xfree, 1);
    for (int l = 0; l < 2; ++l) mbar_init(&hfull[l], EPI_WARPS);
    for (int l = 0; l < 3; ++l) mbar_init(&tfull[l], 1);
    for (int s = 0; s < WSTAGES; ++s) {
      mbar_init(&wfull[s], 1);
      mbar_init(&wempty[s], 1);
    }
    mbar_fence_init();
  }
  for (int c = threadIdx.x; c < 3 * 256; c += THREADS) bias_s[c] = c % 256 < L.n[c / 256 + 1] ? L.bias[c / 256][c % 256] : 0.f;
  // columns past the input width stay zero: the loaders never write them
  for (int c = threadIdx.x; c < (int)(XK * SLICE / 16); c += THREADS) reinterpret_cast<uint4*>(Xs)[c] = make_uint4(0, 0, 0, 0);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = *tslot;
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      // ---- weight slices of every tile ----
      int it = 0;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        for (int l = 0; l < 3 && ok; ++l) {
          const CUtensorMap* map = l == 0 ? &w1 : (l == 1 ? &w2 : &w3);
          const unsigned bytes = (unsigned)umws::npad_of(L.n[l + 1]) * 128u;
          for (int kb = 0; kb < umws::nkb_of(L.kp[l]); ++kb, ++it) {
            const int s = it % WSTAGES, u = it / WSTAGES;
            if (u > 0 && !mbar_wait(&wempty[s], (unsigned)((u - 1) & 1), kWaitPolls)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&wfull[s], bytes);
            umws::tma_load_2d(Ws + (size_t)s * WSTAGE, map, kb * BK, 0, &wfull[s]);
          }
        }
      }
      if (!ok) atomicExch(err, 1);
      for (int j = it > WSTAGES ? it - WSTAGES : 0; j < it; ++j)  // copies still in flight
        (void)mbar_wait(&wfull[j % WSTAGES], (unsigned)((j / WSTAGES) & 1), kWaitPolls);
    }
  } else if (warp == 1) {
    // ---- MMA issue: the whole warp walks the slices, so addresses and descriptors are uniform
    // values (an issue from one lane's registers costs 140 clocks, more than the MMA) ----
    const bool one = elect_one();
    int it = 0, t = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++t) {
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        // layer 1 reads X, layers 2 and 3 what the epilogue leaves in tensor memory
        ok = ok && warp_wait(l == 0 ? xfull : &hfull[l - 1], (unsigned)(t & 1));
        const unsigned acc = tmem + (l < 2 ? 0u : COL_OUT);
        const unsigned id = umws::idesc_bf16(BM, umws::npad_of(L.n[l + 1]));
        const int nkb = umws::nkb_of(L.kp[l]), k16 = (L.kp[l] + 15) / 16;
        for (int kb = 0; kb < nkb && ok; ++kb) {
          const int s = it % WSTAGES, u = it / WSTAGES;
          ok = warp_wait(&wfull[s], (unsigned)(u & 1));
          if (!ok) break;
          ++it;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const unsigned long long ad = umws::sdesc_sw128(smem_u32(Xs) + (unsigned)kb * SLICE);
          const unsigned long long bd = umws::sdesc_sw128(smem_u32(Ws) + (unsigned)s * WSTAGE);
          const unsigned h0 = tmem + COL_H + (unsigned)kb * (BK / 2);
          const int steps = k16 - kb * (BK / 16);
          if (one) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
              if (kk < steps) {
                const unsigned more = kk > 0 || kb > 0 ? 1u : 0u;
                if (l == 0)
                  asm volatile(
                      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(acc),
                      "l"(ad + 2u * kk), "l"(bd + 2u * kk), "r"(id), "r"(more)
                      : "memory");
                else
                  asm volatile(
                      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(acc),
                      "r"(h0 + 8u * kk), "l"(bd + 2u * kk), "r"(id), "r"(more)
                      : "memory");
              }
            }
            commit(&wempty[s]);
          }
          __syncwarp();
        }
        if (ok && one) {
          commit(&tfull[l]);
          if (l == 0) commit(xfree);
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) atomicExch(err, 1);
    for (int j = it > WSTAGES ? it - WSTAGES : 0; j < it; ++j)  // MMAs still in flight
      (void)warp_wait(&wempty[j % WSTAGES], (unsigned)((j / WSTAGES) & 1));
  } else if (warp < 2 + EPI_WARPS) {
    // ---- epilogues: four warps per lane quarter; of a hidden layer each takes one slice of 64
    // columns, of the output every fourth group of 16 ----
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int r = q * 32 + lane;
    const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
    int t = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++t) {
      const long long row = (long long)tile * BM + r;
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        ok = warp_wait(&tfull[l], (unsigned)(t & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned lanes = tmem + ((unsigned)(q * 32) << 16), taddr = lanes + (l < 2 ? 0u : COL_OUT);
        const int n = L.n[l + 1], npad = umws::npad_of(n);
        const int c_first = l < 2 ? 64 * part : 16 * part, c_step = l < 2 ? 16 : 64;
        unsigned v[2][16];  // this group's columns and the next one's, in flight
        if (c_first < npad) tmem_ld16(v[0], taddr + c_first);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int c0 = c_first + g * c_step;
          if (c0 < npad) {
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (g < 3 && c0 + c_step < npad) tmem_ld16(v[(g + 1) & 1], taddr + c0 + c_step);
            const float4* b4 = reinterpret_cast<const float4*>(bias_s + l * 256 + c0);
            float2 x[8];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 b = b4[k];
              const unsigned* a = &v[g & 1][4 * k];
              x[2 * k] = add2(make_float2(__uint_as_float(a[0]), __uint_as_float(a[1])), make_float2(b.x, b.y));
              x[2 * k + 1] = add2(make_float2(__uint_as_float(a[2]), __uint_as_float(a[3])), make_float2(b.z, b.w));
            }
            if (l < 2) {
              unsigned w[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(x[k].x, x[k].y), zero);
                w[k] = *reinterpret_cast<const unsigned*>(&h);
              }
              asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(
                               lanes + COL_H + (unsigned)c0 / 2),
                           "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                           : "memory");
            } else if (n % 4 == 0) {
              // rows of four lanes exchanged, so that four lanes store 64 consecutive bytes of a row
              transpose4(x, lane);
              const long long first = row - (lane & 3);
              const int c = c0 + 4 * (lane & 3);
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (first + k < M && c < n)
                  __stcs(reinterpret_cast<float4*>(Y + (first + k) * n + c),
                         make_float4(x[2 * k].x, x[2 * k].y, x[2 * k + 1].x, x[2 * k + 1].y));
            } else if (row < M) {
              float* o = Y + (size_t)row * n + c0;
#pragma unroll
              for (int k = 0; k < 16; ++k)
                if (c0 + k < n) o[k] = k & 1 ? x[k / 2].y : x[k / 2].x;
            }
          }
        }
        if (l < 2) {
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");  // also after the output of the tile before
          __syncwarp();
          if (lane == 0) arrive(&hfull[l]);
        }
      }
    }
    if (!ok && lane == 0) atomicExch(err, 1);
  } else {
    // ---- X: FLIGHT to 2 FLIGHT pieces of four columns in flight per lane ----
    constexpr int FLIGHT = 4;
    const int w = warp - 2 - EPI_WARPS, nq = L.n[0] / 4;
    const int row0 = (w * 32 + lane) / nq, col0 = (w * 32 + lane) % nq, dr = 32 * LOAD_WARPS / nq, dk = 32 * LOAD_WARPS % nq;
    int t = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++t) {
      if (t > 0 && !warp_wait(xfree, (unsigned)((t - 1) & 1))) {
        if (lane == 0) atomicExch(err, 1);
        break;
      }
      const long long r0 = (long long)tile * BM;
      const int rows = (int)min((long long)BM, M - r0);
      const float4* src = reinterpret_cast<const float4*>(X + r0 * L.n[0]);
      int r = row0, k = col0;  // of the next store; the tile's 16-byte pieces lie one after another
      int e = w * 32 + lane;  // of the next load
      float4 v[2][FLIGHT];
      const auto load = [&](float4 (&d)[FLIGHT]) {
#pragma unroll
        for (int u = 0; u < FLIGHT; ++u, e += 32 * LOAD_WARPS) d[u] = e < rows * nq ? __ldcs(src + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      const auto store = [&](const float4 (&d)[FLIGHT]) {
#pragma unroll
        for (int u = 0; u < FLIGHT; ++u) {
          if (r < BM) {
            const __nv_bfloat162 a = __floats2bfloat162_rn(d[u].x, d[u].y), b = __floats2bfloat162_rn(d[u].z, d[u].w);
            *reinterpret_cast<uint2*>(Xs + chunk_of(r, 4 * k & ~7) + (k & 1) * 8) =
                make_uint2(*reinterpret_cast<const unsigned*>(&a), *reinterpret_cast<const unsigned*>(&b));
          }
          r += dr;
          k += dk;
          if (k >= nq) {
            k -= nq;
            ++r;
          }
        }
      };
      load(v[0]);
      while (r < BM) {
        load(v[1]);
        store(v[0]);
        load(v[0]);
        store(v[1]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) arrive(xfull);
      if (w == 0 && lane == 0 && tile + (int)gridDim.x < ntiles) {  // the next tile's rows on their way to L2
        const long long next = r0 + (long long)gridDim.x * BM;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(X + next * L.n[0]),
                     "r"((unsigned)min((long long)BM, M - next) * L.n[0] * 4u)
                     : "memory");
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(umws::TMEM_COLS) : "memory");
}

}  // namespace mlpf
}  // namespace frk
