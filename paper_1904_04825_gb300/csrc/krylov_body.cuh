// The vector phases of an Arnoldi iteration, shared by the per-phase kernels
// (krylov.cu) and the GMRES cycle kernel (cycle.cuh): block bid of nblk handles
// the same rows in the same order in both, so their sums agree bit for bit.
#pragma once

#include "device.cuh"

namespace frk {

// this thread's share of ||x||^2: one FMA chain in row order, eight loads in
// flight (with one, 16.8 M rows ran at a tenth of HBM's rate)
__device__ __forceinline__ double sumsq_rows(const double* x, long long n, int bid, int nblk) {
  const long long S = (long long)nblk * blockDim.x;
  long long i = (long long)bid * blockDim.x + threadIdx.x;
  double ss = 0.0;
  for (; i + 7 * S < n; i += 8 * S) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = x[i + u * S];
#pragma unroll
    for (int u = 0; u < 8; ++u) ss = fma(v[u], v[u], ss);
  }
  for (; i < n; i += S) ss = fma(x[i], x[i], ss);
  return ss;
}

// One sweep over the rows accumulating NC dot products against w; the
// basis pointers are resolved outside the row loop so every row costs
// exactly NC fused multiply-adds on the FP64 pipe.  UR rows are in flight per
// thread (NC x UR independent accumulation chains hide the FMA latency).
template <int NC>
__device__ __forceinline__ void dots_chunk(const double* const* ptr, const double* w,
                                           long long n, double* acc, int bid, int nblk) {
  constexpr int UR = NC >= 8 ? 1 : (NC >= 4 ? 2 : 4);
  double a[NC][UR];
#pragma unroll
  for (int i = 0; i < NC; ++i)
#pragma unroll
    for (int u = 0; u < UR; ++u) a[i][u] = 0.0;
  const long long S = (long long)nblk * blockDim.x;
  for (long long r0 = (long long)bid * blockDim.x + threadIdx.x; r0 < n; r0 += UR * S) {
    double wr[UR];
#pragma unroll
    for (int u = 0; u < UR; ++u) wr[u] = (r0 + u * S < n) ? w[r0 + u * S] : 0.0;
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
      for (int u = 0; u < UR; ++u)
        if (r0 + u * S < n) a[i][u] = fma(ptr[i][r0 + u * S], wr[u], a[i][u]);
  }
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    double s = a[i][0];
#pragma unroll
    for (int u = 1; u < UR; ++u) s += a[i][u];
    acc[i] = s;
  }
}

// Block bid's partials of <V_i, w> for i < nvec, and of <w, w> behind them when
// total = nvec + 1, in chunks of up to 8 values per sweep; the warps' sums of all
// chunks meet once at the end, so a chunk's loads need not wait for the one before.
// Blocks of kThreads threads.
__device__ __forceinline__ void dots_partials(const double* V, long long ldv, int nvec, const double* w, long long n,
                                              int total, const Reduce& red, int bid, int nblk) {
  __shared__ double sred[kMaxVec][kThreads / 32 + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  static_assert(kThreads == 256, "eight warps");
  for (int c0 = 0; c0 < total; c0 += 8) {
    const int nc = min(8, total - c0);
    const double* ptr[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int idx = c0 + i;
      ptr[i] = idx < nvec ? V + (size_t)idx * ldv : w;
    }
    double acc[8];
    switch (nc) {
      case 1: dots_chunk<1>(ptr, w, n, acc, bid, nblk); break;
      case 2: dots_chunk<2>(ptr, w, n, acc, bid, nblk); break;
      case 3: dots_chunk<3>(ptr, w, n, acc, bid, nblk); break;
      case 4: dots_chunk<4>(ptr, w, n, acc, bid, nblk); break;
      case 5: dots_chunk<5>(ptr, w, n, acc, bid, nblk); break;
      case 6: dots_chunk<6>(ptr, w, n, acc, bid, nblk); break;
      case 7: dots_chunk<7>(ptr, w, n, acc, bid, nblk); break;
      default: dots_chunk<8>(ptr, w, n, acc, bid, nblk); break;
    }
    // Warp sums of the (up to) 8 values by recursive halving: each exchange
    // sends half of the values still held to the partner lane and keeps the
    // other half, so lane l ends with the warp sum of value
    // 4 b4 + 2 b3 + b2 (b = bits of l) after 9 additions instead of 8 x 5.
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i >= nc) acc[i] = 0.0;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double send = b4 ? acc[q] : acc[q + 4];
      const double keep = b4 ? acc[q + 4] : acc[q];
      acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double send = b3 ? acc[q] : acc[q + 2];
      const double keep = b3 ? acc[q + 2] : acc[q];
      acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    {
      const double send = b2 ? acc[0] : acc[1];
      const double keep = b2 ? acc[1] : acc[0];
      acc[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    const int vi = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
    if ((lane & 3) == 0 && vi < nc) sred[c0 + vi][wid] = acc[0];
  }
  __syncthreads();
  if ((int)threadIdx.x < total) {
    const double* t = sred[threadIdx.x];
    red.value(threadIdx.x)[bid] = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
  }
  __syncthreads();
}

// out[i] = <V_i, w> for i < nvec, and out[nvec] = <w, w> when with_self.  Skipped
// when the cycle is done or when `gate` points at a zero flag.
__device__ __forceinline__ void dots_body(const double* V, long long ldv, int nvec, const double* w, long long n,
                                          double* out, int with_self, const Reduce& red, const int* done,
                                          const int* gate, int bid, int nblk) {
  if ((done && *done) || (gate && !*gate)) return;
  const int total = nvec + (with_self ? 1 : 0);
  dots_partials(V, ldv, nvec, w, n, total, red, bid, nblk);
  if (last_block(red.counter, nblk)) finish_sums(red, total, out, nblk);
}

// w -= sum_i h_i V_i as one FMA chain per row (exactly nvec FP64 FMAs); optional sum of
// squares of the new w.  With `self2` (the first Gram-Schmidt pass) the last
// block also decides whether iteration j needs the second pass: it does when
// ||w_new|| < eta ||w_old|| (the test of Daniel, Gragg, Kaufman and Stewart;
// one classical pass leaves an orthogonality error of about
// u ||w_old|| / ||w_new||, so eta = 1/64 keeps it below ~64 u), recorded in
// rflag[j]; otherwise h2 is cleared.
struct Reorth {
  const double* self2;  // ||w||^2 before the first pass, or nullptr
  double eta2;          // second pass when ||w_new||^2 < eta2 ||w_old||^2
  int* rflag;           // &rflag[j]
  double* h2;
};

// block bid's rows; returns the thread's share of the new ||w||^2
__device__ __forceinline__ double update_rows(double* w, const double* V, long long ldv, int nvec,
                                              const double* neg_h, long long n, int bid, int nblk) {
  // four rows per thread in flight: four independent FMA chains of length nvec
  constexpr int UR = 4;
  double ss[UR] = {0.0, 0.0, 0.0, 0.0};
  const long long S = (long long)nblk * blockDim.x;
  if (n <= S) {  // one row per thread: the loads of 16 vectors in flight instead of four rows'
    const long long r = (long long)bid * blockDim.x + threadIdx.x;
    if (r >= n) return 0.0;
    double v = w[r];
    for (int i0 = 0; i0 < nvec; i0 += 16) {
      double x[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) x[u] = i0 + u < nvec ? V[(i0 + u) * ldv + r] : 0.0;
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (i0 + u < nvec) v = fma(neg_h[i0 + u], x[u], v);
    }
    w[r] = v;
    return v * v;
  }
  for (long long r0 = (long long)bid * blockDim.x + threadIdx.x; r0 < n; r0 += UR * S) {
    double v[UR];
#pragma unroll
    for (int u = 0; u < UR; ++u) v[u] = (r0 + u * S < n) ? w[r0 + u * S] : 0.0;
    for (int i = 0; i < nvec; ++i) {
      const double hi = neg_h[i];
      const double* Vi = V + i * ldv;
#pragma unroll
      for (int u = 0; u < UR; ++u)
        if (r0 + u * S < n) v[u] = fma(hi, Vi[r0 + u * S], v[u]);
    }
#pragma unroll
    for (int u = 0; u < UR; ++u) {
      if (r0 + u * S < n) {
        w[r0 + u * S] = v[u];
        ss[u] = fma(v[u], v[u], ss[u]);
      }
    }
  }
  return (ss[0] + ss[1]) + (ss[2] + ss[3]);
}

__device__ __forceinline__ void update_body(double* w, const double* V, long long ldv, int nvec, const double* h,
                                            long long n, double* sumsq, const Reduce& red, const int* done,
                                            const int* gate, const Reorth& ro, int bid, int nblk) {
  __shared__ double sh[32];
  __shared__ double hs[kMaxVec];
  if ((done && *done) || (gate && !*gate)) return;
  if (threadIdx.x < nvec) hs[threadIdx.x] = -h[threadIdx.x];
  __syncthreads();
  const double bs = block_sum(update_rows(w, V, ldv, nvec, hs, n, bid, nblk), sh);
  if (threadIdx.x == 0) red.value(0)[bid] = bs;
  if (last_block(red.counter, nblk)) {
    finish_sums(red, 1, sumsq, nblk);
    if (ro.self2 && threadIdx.x == 0) {
      const int need = (*sumsq < ro.eta2 * *ro.self2) ? 1 : 0;
      *ro.rflag = need;
      if (!need)
        for (int q = 0; q < nvec; ++q) ro.h2[q] = 0.0;
    }
  }
}

// Hessenberg column j, Givens rotations, residual estimate, convergence.
// One warp: the lanes bring the column's Gram-Schmidt coefficients and the
// earlier rotations into shared memory together (one round of independent
// loads instead of a chain of dependent ones), lane 0 applies the rotations
// in order, and the lanes write the column back.
__device__ __forceinline__ void givens_body(const GmresDev& gd, int j, const double* nw2) {
  __shared__ double hs[kMaxVec + 1], cs_s[kMaxVec], sn_s[kMaxVec];
  if (*gd.done) return;
  const int lane = threadIdx.x & 31;
  for (int i = lane; i <= j; i += 32) hs[i] = gd.h1[i] + gd.h2[i];
  for (int i = lane; i < j; i += 32) {
    cs_s[i] = gd.cs[i];
    sn_s[i] = gd.sn[i];
  }
  __syncwarp();
  if (lane == 0) {
    const double hn = sqrt(*nw2);
    hs[j + 1] = hn;
    for (int i = 0; i < j; ++i) {
      const double t = cs_s[i] * hs[i] + sn_s[i] * hs[i + 1];
      hs[i + 1] = -sn_s[i] * hs[i] + cs_s[i] * hs[i + 1];
      hs[i] = t;
    }
    const double den2 = fma(hs[j], hs[j], hs[j + 1] * hs[j + 1]);
    double den, c, s;
    if (den2 > 1e-280 && den2 < 1e280) {  // no scaling needed (hypot is most of this lane's chain)
      den = sqrt(den2);
      const double r = 1.0 / den;
      c = hs[j] * r;
      s = hs[j + 1] * r;
    } else {
      den = hypot(hs[j], hs[j + 1]);
      c = den > 0.0 ? hs[j] / den : 1.0;
      s = den > 0.0 ? hs[j + 1] / den : 0.0;
    }
    gd.cs[j] = c;
    gd.sn[j] = s;
    hs[j] = den;
    hs[j + 1] = 0.0;
    gd.g[j + 1] = -s * gd.g[j];
    gd.g[j] = c * gd.g[j];
    *gd.k = j + 1;
    const double res = fabs(gd.g[j + 1]);
    *gd.res = res;
    gd.invh[j + 1] = hn > 0.0 ? 1.0 / hn : 0.0;
    if (res <= *gd.target || hn == 0.0 || !(res == res)) *gd.done = 1;
  }
  __syncwarp();
  double* Hj = gd.H + (size_t)j * gd.ldh;
  for (int i = lane; i <= j + 1; i += 32) Hj[i] = hs[i];
}

constexpr int kTriangle = kMaxVec * (kMaxVec - 1) / 2;  // packed triangle of up to kMaxVec - 1 columns

// y = H(0:k,0:k)^{-1} g(0:k) into ys (shared, k values) by the whole block.  The
// triangle comes into shared memory at once (Hs, kTriangle values); then one warp
// settles the unknowns from the last up and subtracts each from all rows above
// it together (one lane doing that row by row took 24 us at k = 20).
__device__ __forceinline__ void backsub(const GmresDev& gd, int k, double* Hs, double* ys) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int l = wid; l < k; l += nw)
    for (int i = lane; i <= l; i += 32) Hs[l * (l + 1) / 2 + i] = gd.H[(size_t)l * gd.ldh + i];
  for (int i = threadIdx.x; i < k; i += blockDim.x) ys[i] = gd.g[i];
  __syncthreads();
  if (wid == 0) {
    for (int l = k - 1; l >= 0; --l) {
      const double* Hl = Hs + l * (l + 1) / 2;
      const double y = ys[l] / Hl[l];
      __syncwarp();
      for (int i = lane; i < l; i += 32) ys[i] = fma(-Hl[i], y, ys[i]);
      if (lane == 0) ys[l] = y;
      __syncwarp();
    }
  }
  __syncthreads();
}

}  // namespace frk
