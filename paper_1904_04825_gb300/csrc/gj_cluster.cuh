// Gauss-Jordan inversion of element blocks too large for one SM's shared
// memory (the element-Jacobi preconditioner of Sec. 4.5 for 3D degree 3:
// 5 (p+1)^3 = 320 rows, 400 KB in FP32), split over a cluster of two CTAs.
//
// CTA r of the cluster holds columns [r NB/2, (r+1) NB/2) of the FP32 matrix
// in its shared memory (row stride NB/2 + 1).  The pivots are taken in
// panels of BW = 16 columns:
//  * a panel's holder factorises it in registers, one row per thread of the
//    panel warps: for each column c the pivot row is the unused row of largest
//    |M[r][c]| (rows stay in place, pr[c] = r is recorded), found by a warp
//    maximum and one shared exchange, two barriers a pivot, and the elimination
//    is applied to the panel's columns;
//  * U = (panel columns after the panel) - (unit vectors of the pivot rows),
//    NB x BW, goes to the shared memory of both CTAs (distributed shared
//    memory), with the panel's pivot rows;
//  * every other column takes x <- x + U x_P, x_P the pivot rows' entries of x
//    before the panel (a rank-BW update on the CUDA cores, FP32).  The panel
//    warps of the next panel's holder do that for that panel alone and go on to
//    factorise it while the update warps bring the rest up to date, so the serial
//    pivot chain runs behind the updates;
//  * a cluster barrier ends the updates, then the holder publishes the next U and
//    a second one makes it visible.
// Every entry sees the same operations in the same order as without the overlap.
// Bound: the pivot chain (two block barriers, a maximum, a reciprocal per pivot).
// 4096 blocks of 320 rows: 15.2 ms; 23.1 ms when each panel was factorised while
// both CTAs' updates waited, with five-step shuffles for each maximum.
// The result is the inverse with permuted rows and columns:
// inverse(a, b) = M[pr[a]][c] with pr[c] = b.
#pragma once

#include <cooperative_groups.h>

#include "device.cuh"

namespace frk {
namespace gjcl {

constexpr int CL = 2;         // CTAs per cluster
constexpr int BW = 16;        // panel width
constexpr int PANEL = 320;        // panel threads: one row each
constexpr int UPDATE = 320;       // update threads
constexpr int THREADS = PANEL + UPDATE;

template <int NB>
struct Shape {
  static_assert(NB % (CL * 32) == 0, "each CTA's columns are whole warps of lanes");
  static constexpr int CW = NB / CL;         // columns per CTA
  static constexpr int LDM = CW + 1;         // row stride of M (conflict-free column reads)
  static constexpr int QN = CW / 32;         // columns per lane in the update
  static_assert(NB == PANEL, "the panel factorisation keeps one row per thread");
  // bytes: M, U, the next panel's x_P, pr (int), rows (int), pivot row (16-byte
  // aligned), per-warp pivot candidates
  static constexpr size_t OFF_U = (size_t)NB * LDM * 4;
  static constexpr size_t OFF_XP = OFF_U + (size_t)NB * BW * 4;
  static constexpr size_t OFF_SROW = OFF_XP + (size_t)BW * BW * 4;
  static constexpr size_t OFF_CAND = OFF_SROW + BW * 4;
  static constexpr size_t OFF_PR = OFF_CAND + 32 * 8;
  static constexpr size_t OFF_ROWS = OFF_PR + (size_t)NB * 4;
  static constexpr size_t BYTES = (OFF_ROWS + BW * 4 + 15) / 16 * 16;
};

__device__ __forceinline__ void group_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The pivots of one panel: thread i of the panel warps holds row i in pv.
// prow[k] receives the pivot rows; usd: the row is a pivot row already.
__device__ __forceinline__ void factorise(float pv[BW], bool& usd, int i, float* srow, uint2* cand, int* prow) {
  constexpr int NW = PANEL / 32;
  const int lane = i & 31, warp = i >> 5;
#pragma unroll
  for (int k = 0; k < BW; ++k) {
    // the unused row of largest |M[r][c]| (a NaN ranks as an infinity), the
    // lowest row among equals: magnitudes order as their bit patterns
    unsigned key = 0u;
    if (!usd) {
      const unsigned m = __float_as_uint(pv[k]) & 0x7fffffffu;
      key = (m > 0x7f800000u ? 0x7f800000u : m) + 1u;
    }
    const unsigned best = __reduce_max_sync(0xffffffffu, key);
    const unsigned who = __ballot_sync(0xffffffffu, key == best);
    if (lane == 0) cand[warp] = make_uint2(best, (unsigned)(warp * 32 + __ffs(who) - 1));
    group_barrier(1, PANEL);
    const uint2 c = lane < NW ? cand[lane] : make_uint2(0u, 0u);
    const unsigned top = __reduce_max_sync(0xffffffffu, c.x);
    const unsigned from = __ballot_sync(0xffffffffu, c.x == top);
    const int r = (int)__shfl_sync(0xffffffffu, c.y, __ffs(from) - 1);
    const float m = pv[k];  // this row's entry in the pivot column
    if (i == r) {
      const float ip = 1.f / m;
#pragma unroll
      for (int t = 0; t < BW; ++t) srow[t] = (t == k ? 1.f : pv[t]) * ip;
      prow[k] = r;
      usd = true;
    }
    group_barrier(1, PANEL);
    const float4* s4 = reinterpret_cast<const float4*>(srow);
#pragma unroll
    for (int t4 = 0; t4 < BW / 4; ++t4) {
      const float4 v = s4[t4];
      const float sr[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int t = 4 * t4 + q;
        pv[t] = i == r ? sr[q] : (t == k ? 0.f : pv[t]) - m * sr[q];
      }
    }
  }
}

// M[:, j] += U x_P[:, j] for the columns j = lane + 32 q, Q0 <= q < Q1, outside the
// panel at local column lc and the next one at nl, by warp wi's rpw rows; `threads`
// update threads take part
template <int NB, int Q0, int Q1>
__device__ __forceinline__ void update_columns(float* M, const float* U, const int* rows, int lane, int wi, int rpw, int lc,
                                               int nl, int threads) {
  constexpr int LDM = Shape<NB>::LDM, Q = Q1 - Q0;
  float x[BW][Q];
  bool keep[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = lane + 32 * (Q0 + q);
    keep[q] = !(j >= lc && j < lc + BW) && !(j >= nl && j < nl + BW);
#pragma unroll
    for (int k = 0; k < BW; ++k) x[k][q] = M[rows[k] * LDM + j];  // before any row of these columns changes
  }
  group_barrier(2, threads);
  for (int i = wi * rpw; i < (wi + 1) * rpw; ++i) {
    const float4* ui = reinterpret_cast<const float4*>(U + i * BW);
    float acc[Q] = {};
#pragma unroll
    for (int k4 = 0; k4 < BW / 4; ++k4) {
      const float4 v = ui[k4];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        acc[q] = fmaf(v.x, x[4 * k4][q], acc[q]);
        acc[q] = fmaf(v.y, x[4 * k4 + 1][q], acc[q]);
        acc[q] = fmaf(v.z, x[4 * k4 + 2][q], acc[q]);
        acc[q] = fmaf(v.w, x[4 * k4 + 3][q], acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (keep[q]) M[i * LDM + lane + 32 * (Q0 + q)] += acc[q];
  }
}

// Invert element blocks b = 0 .. (gridDim.x / CL) - 1 of the FP64 staging
// mst (column-major per element: mst[b][c][row]) into blocks + (e0 + b) NB^2
// (column-major: Minv[k NB + i] = inverse(i, k)), adding dshift to the
// diagonal first.  Launched with THREADS threads and Shape<NB>::BYTES of
// dynamic shared memory per CTA, clusters of CL CTAs along x.
template <int NB, typename S, typename Store>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(THREADS)
    k_invert_cluster(const double* __restrict__ mst, S* __restrict__ blocks, long long e0, double dshift) {
  namespace cg = cooperative_groups;
  using Sh = Shape<NB>;
  constexpr int CW = Sh::CW, LDM = Sh::LDM, QN = Sh::QN;
  extern __shared__ __align__(16) unsigned char smem_cl[];
  float* M = reinterpret_cast<float*>(smem_cl);
  float* U = reinterpret_cast<float*>(smem_cl + Sh::OFF_U);
  float* xp = reinterpret_cast<float*>(smem_cl + Sh::OFF_XP);
  float* srow = reinterpret_cast<float*>(smem_cl + Sh::OFF_SROW);
  uint2* cand = reinterpret_cast<uint2*>(smem_cl + Sh::OFF_CAND);
  int* pr = reinterpret_cast<int*>(smem_cl + Sh::OFF_PR);
  int* rows = reinterpret_cast<int*>(smem_cl + Sh::OFF_ROWS);

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31;
  const long long b = blockIdx.x / CL;
  const int col0 = rank * CW;
  const double* src = mst + b * (long long)NB * NB;
  for (int idx = tid; idx < CW * NB; idx += THREADS) {
    const int lc = idx / NB, i = idx - lc * NB;
    const double v = src[(long long)(col0 + lc) * NB + i];
    M[i * LDM + lc] = (float)(i == col0 + lc ? v + dshift : v);
  }
  float* peerU = cluster.map_shared_rank(U, rank ^ 1);
  int* peerRows = cluster.map_shared_rank(rows, rank ^ 1);
  cluster.sync();  // both CTAs' shared memory is set up before any remote write

  const bool panel_warp = tid < PANEL;
  bool usd = false;  // panel threads: row tid is a pivot row of an earlier panel
  float pv[BW];      // panel threads: row tid of the panel being factorised
  // the panel at local column lc back into M; U and the pivot rows to both CTAs
  // (the pivot rows of the panel are in pr[c0 ..] of this CTA)
  auto publish = [&](int lc, int c0) {
    const int i = tid;
    float4* u4 = reinterpret_cast<float4*>(U + i * BW);
    float4* p4 = reinterpret_cast<float4*>(peerU + i * BW);
#pragma unroll
    for (int t4 = 0; t4 < BW / 4; ++t4) {
      float u[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int t = 4 * t4 + q;
        M[i * LDM + lc + t] = pv[t];
        u[q] = pv[t] - (i == pr[c0 + t] ? 1.f : 0.f);
      }
      const float4 v = make_float4(u[0], u[1], u[2], u[3]);
      u4[t4] = v;
      p4[t4] = v;
    }
    if (i < BW) {
      rows[i] = pr[c0 + i];
      peerRows[i] = pr[c0 + i];
    }
  };
  if (rank == 0 && panel_warp) {
#pragma unroll
    for (int t = 0; t < BW; ++t) pv[t] = M[tid * LDM + t];
    factorise(pv, usd, tid, srow, cand, pr);
    group_barrier(1, PANEL);  // pr is complete
    publish(0, 0);
  }
  for (int c0 = 0; c0 < NB; c0 += BW) {
    cluster.sync();  // U and the pivot rows of panel c0 are visible in both CTAs
    const int lc0 = c0 - col0;                    // this panel's local columns (if here)
    const int n0 = c0 + BW, nl0 = n0 - col0;      // the next panel's
    const bool next_here = n0 < NB && n0 / CW == rank;
    if (panel_warp) {
      if (tid < BW) pr[c0 + tid] = rows[tid];
#pragma unroll
      for (int k = 0; k < BW; ++k) usd = usd || rows[k] == tid;
    }
    if (next_here && panel_warp) {
      // the next panel's columns first, in registers, and its pivots
      for (int q = tid; q < BW * BW; q += PANEL) xp[q] = M[rows[q / BW] * LDM + nl0 + q % BW];
      group_barrier(1, PANEL);
      const float4* ui = reinterpret_cast<const float4*>(U + tid * BW);
      float u[BW];
#pragma unroll
      for (int k4 = 0; k4 < BW / 4; ++k4) {
        const float4 v = ui[k4];
        u[4 * k4] = v.x;
        u[4 * k4 + 1] = v.y;
        u[4 * k4 + 2] = v.z;
        u[4 * k4 + 3] = v.w;
      }
      const float4* x4 = reinterpret_cast<const float4*>(xp);
#pragma unroll
      for (int t4 = 0; t4 < BW / 4; ++t4) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < BW; ++k) {
          const float4 x = x4[k * (BW / 4) + t4];
          acc[0] = fmaf(u[k], x.x, acc[0]);
          acc[1] = fmaf(u[k], x.y, acc[1]);
          acc[2] = fmaf(u[k], x.z, acc[2]);
          acc[3] = fmaf(u[k], x.w, acc[3]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) pv[4 * t4 + q] = M[tid * LDM + nl0 + 4 * t4 + q] + acc[q];
      }
      factorise(pv, usd, tid, srow, cand, pr + n0);
      group_barrier(1, PANEL);  // pr is complete
    } else {
      // M[:, j] += U x_P[:, j] for this CTA's other columns: the update warps, and
      // the panel warps too where they have no panel
      const int first = next_here ? PANEL : 0, wi = (tid - first) >> 5;
      const int nw = (THREADS - first) / 32, rpw = NB / nw;
      static_assert(NB % (THREADS / 32) == 0 && NB % (UPDATE / 32) == 0, "rows split evenly over the warps");
      // in two passes over the lane's columns, so that x_P stays in registers
      update_columns<NB, 0, (QN + 1) / 2>(M, U, rows, lane, wi, rpw, lc0, next_here ? nl0 : -BW, THREADS - first);
      update_columns<NB, (QN + 1) / 2, QN>(M, U, rows, lane, wi, rpw, lc0, next_here ? nl0 : -BW, THREADS - first);
    }
    if (n0 < NB) {
      cluster.sync();  // every CTA is done with U before the next panel's overwrites it
      if (next_here && panel_warp) publish(nl0, n0);
    }
  }
  cluster.sync();  // neither CTA leaves while the other may still write to it
  // ---- store: inverse(ii, kk) = M[pr[ii]][c] for this CTA's columns c, kk = pr[c] ----
  S* out = blocks + (e0 + b) * (long long)NB * NB;
  for (int idx = tid; idx < CW * NB; idx += THREADS) {
    const int lc = idx / NB, ii = idx - lc * NB;
    out[(long long)pr[col0 + lc] * NB + ii] = Store::to(M[pr[ii] * LDM + lc]);
  }
}

}  // namespace gjcl
}  // namespace frk
