// Gauss-Jordan inversion of one FP64 element block (the element-Jacobi
// preconditioner of Sec. 4.5) with the trailing updates on the integer units.
//
// In-place Gauss-Jordan with partial pivoting in panels of BW = 16 columns, like
// gj_tc.cuh: a panel's pivots are found and eliminated on the panel's
// columns alone in FP64 (the rows in registers, TPR threads a row), rows stay in
// place (pr[c] = the pivot row of column c); then every other column takes
//   M[:, j] = (0 in the pivot rows, M[:, j] in the others) + U x_P[:, j],
// U the panel after its pivots and x_P the pivot rows before them, a rank-16 update
// whose sums of 16 products are formed as integers (fx.cuh) and added to M with one
// rounding.  A pivot row is formed from the products alone: as M + (U - 1) x_P, a
// difference of nearly equal numbers where the pivot is large, it kept only the
// absolute accuracy of M, and one variable of the inverse lost 8 digits in SI units.
// An operand keeps 57 bits below its group's largest value (groups: a row of U, a
// column of x_P), so term k of the sums is scaled by 2^t_k, which leaves the products
// as they are and evens the groups: t_k the largest exponent of row k of x_P, each
// column's entries taken relative to its largest.  That takes out whatever units the
// rows and columns have.  Worst variable of M^-1 r against the exact inverse, by
// elimination one pivot at a time in FP64 / here: unit scaling 7e-16 / 4e-16, cells of
// 1e-4 width 2e-14 / 2e-14, SI units (p = 2) 5e-13 / 2e-13.
// The result is the inverse with permuted rows and columns:
// inverse(a, b) = M[pr[a]][ipr[b]].
//
// Bound: FP64 issue.  Rank-1 elimination takes NB^3 FP64 multiply-adds; here
// NB^2 BW of them stay in the panels, and an updated entry costs 2 FP64
// operations per panel instead of 16: at NB = 64 90 thousand instead of 262
// thousand.  Formation and inversion of the 25,600 blocks of the 160 x 160, p = 3
// mesh: 9.2 ms, 17.8 ms by rank-1 elimination in shared memory (five
// barriers and an integer division per entry and pivot).  Panels of 8 or 32
// columns would put more into the updates' roundings or the panels.
#pragma once

#include "fx.cuh"

namespace frk {
namespace gjfx {

constexpr int BW = 16;

template <int NB, int THREADS>
struct Shape {
  static constexpr int TPR = 2 * NB <= THREADS ? 2 : 1;  // threads per row of a panel
  static constexpr int CPT = BW / TPR;                   // panel columns per thread
  static constexpr int COLS = (NB + 1) / 2 * 2;          // X columns, whole pairs
  static constexpr int ROWS = (NB + 3) / 4 * 4;          // U rows, whole quadruples
  static_assert(NB * TPR <= THREADS, "a thread per row");
  // scratch: U [BW][ROWS], X [BW][COLS] (int2, 16-byte aligned), exponents, the
  // pivot column and scaled pivot row, candidates per warp, pivot rows, the terms'
  // scales t_k, inverse permutation
  static constexpr size_t OFF_U = 0;
  static constexpr size_t OFF_X = OFF_U + (size_t)BW * ROWS * 8;
  static constexpr size_t OFF_COL = OFF_X + (size_t)BW * COLS * 8;
  static constexpr size_t OFF_SROW = OFF_COL + (size_t)NB * 16;  // two pivot columns in turn
  static constexpr size_t OFF_EU = OFF_SROW + (BW + 2) * 8;  // pivot row, 1 / pivot
  static constexpr size_t OFF_EX = OFF_EU + (size_t)ROWS * 4;
  static constexpr size_t OFF_CAND = OFF_EX + (size_t)COLS * 4;
  static constexpr size_t OFF_ROWS = OFF_CAND + 16 * 8;
  static constexpr size_t OFF_T = OFF_ROWS + BW * 4;
  static constexpr size_t OFF_IPR = OFF_T + BW * 4;
  static constexpr size_t BYTES = (OFF_IPR + (size_t)NB * 4 + 15) / 16 * 16;
};

// Invert the NB x NB matrix M (row stride LD, shared memory) in place into the
// permuted form; pr receives the pivot rows, scratch (16-byte aligned) the rest
// with ipr at scratch + OFF_IPR.  The whole CTA of THREADS threads.
template <int NB, int LD, int THREADS>
__device__ void invert(double* M, int* pr, unsigned char* scratch) {
  using Sh = Shape<NB, THREADS>;
  constexpr int TPR = Sh::TPR, CPT = Sh::CPT, ROWS = Sh::ROWS, COLS = Sh::COLS, NW = THREADS / 32;
  int2* U = reinterpret_cast<int2*>(scratch + Sh::OFF_U);
  int2* X = reinterpret_cast<int2*>(scratch + Sh::OFF_X);
  double* col = reinterpret_cast<double*>(scratch + Sh::OFF_COL);
  double* srow = reinterpret_cast<double*>(scratch + Sh::OFF_SROW);
  int* eU = reinterpret_cast<int*>(scratch + Sh::OFF_EU);
  int* eX = reinterpret_cast<int*>(scratch + Sh::OFF_EX);
  uint2* cand = reinterpret_cast<uint2*>(scratch + Sh::OFF_CAND);
  int* rows = reinterpret_cast<int*>(scratch + Sh::OFF_ROWS);
  int* ts = reinterpret_cast<int*>(scratch + Sh::OFF_T);
  int* ipr = reinterpret_cast<int*>(scratch + Sh::OFF_IPR);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = tid / TPR, half = tid % TPR;  // this thread's row and columns [half CPT, ...) of a panel
  const bool mine = row < NB;
  bool used = false;
  if (mine && half == 0) ipr[row] = 0;
  for (int i = tid; i < BW * ROWS; i += THREADS) U[i] = make_int2(0, 0);
  for (int i = tid; i < BW * COLS; i += THREADS) X[i] = make_int2(0, 0);
  __syncthreads();

  for (int c0 = 0; c0 < NB; c0 += BW) {
    const int kb = NB - c0 < BW ? NB - c0 : BW;
    if (tid < BW) ts[tid] = fx::kNone;
    // ---- the panel's pivots ----
    bool pivot = false;  // this row is one of them
    double pv[CPT];
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      const int c = half * CPT + t;
      pv[t] = mine && c < kb ? M[row * LD + c0 + c] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < BW; ++k) {
      if (k >= kb) break;
      const int kh = k / CPT, kt = k % CPT;
      double* pc = col + (k & 1) * NB;
      // the unused row of largest |entry|, by its upper 31 bits (2^-20 relative);
      // a NaN ranks above everything, the lowest row among equals
      unsigned key = 0u;
      if (mine && half == kh) {
        pc[row] = pv[kt];
        if (!used) key = ((unsigned)__double2hiint(pv[kt]) & 0x7fffffffu) + 1u;
      }
      const unsigned best = __reduce_max_sync(0xffffffffu, key);
      const unsigned who = __ballot_sync(0xffffffffu, key == best);
      if (lane == 0) cand[warp] = make_uint2(best, (unsigned)((warp * 32 + __ffs(who) - 1) / TPR));
      __syncthreads();
      uint2 b = cand[0];
#pragma unroll
      for (int w = 1; w < NW; ++w) {
        const uint2 o = cand[w];
        if (o.x > b.x) b = o;
      }
      const int r = (int)b.y;
      if (row == r) {
#pragma unroll
        for (int t = 0; t < CPT; ++t) srow[half * CPT + t] = half == kh && t == kt ? 1.0 : pv[t];
        used = pivot = true;
        if (half == 0) {
          srow[BW] = rcp_fast(pc[r]);
          pr[c0 + k] = r;
          ipr[r] = c0 + k;
          rows[k] = r;
        }
      }
      __syncthreads();
      if (mine) {
        // the pivot row times 1 / pivot, the others minus their entry times that:
        // one multiply-add either way, and no warp runs ahead for one row
        const double ip = srow[BW], c = pc[row];
        const double f = row == r ? ip : -c * ip;
        const double2* s2 = reinterpret_cast<const double2*>(srow + half * CPT);
#pragma unroll
        for (int t = 0; t < CPT; t += 2) {
          const double2 v = s2[t / 2];
          pv[t] = fma(f, v.x, row == r || (half == kh && t == kt) ? 0.0 : pv[t]);
          pv[t + 1] = fma(f, v.y, row == r || (half == kh && t + 1 == kt) ? 0.0 : pv[t + 1]);
        }
      }
    }
    // ---- the panel back into M; the scales of the terms from x_P ----
    if (mine) {
#pragma unroll
      for (int t = 0; t < CPT; ++t)
        if (half * CPT + t < kb) M[row * LD + c0 + half * CPT + t] = pv[t];
        else pv[t] = 0.0;
    }
    const bool other = tid < NB && !(tid >= c0 && tid < c0 + kb);  // this thread's column of x_P
    if (warp * 32 < NB) {
      int ex[BW], top = 0, best = fx::kNone;
#pragma unroll
      for (int k = 0; k < BW; ++k) {
        ex[k] = other && k < kb ? fx::exponent_of(M[rows[k] * LD + tid], 0) : fx::kNone;
        top = max(top, ex[k]);
      }
#pragma unroll
      for (int k = 0; k < BW; ++k) {
        const int m = __reduce_max_sync(0xffffffffu, ex[k] - top);
        if (lane == k) best = m;
      }
      // (a row of zeros stays near kNone, and its column of U becomes zero too)
      if (lane < BW) atomicMax(ts + lane, best);
    }
    __syncthreads();
    // ---- U and x_P as integers ----
    int ep = fx::kNone;  // largest exponent of the row's U, taken over its threads by whole warps
    int tk[CPT];
#pragma unroll
    for (int t = 0; t < CPT; ++t) {
      tk[t] = ts[half * CPT + t];
      if (mine) ep = max(ep, fx::exponent_of(pv[t], tk[t]));
    }
    if (TPR == 2) ep = max(ep, __shfl_xor_sync(0xffffffffu, ep, 1));
    if (mine) {
      if (half == 0) eU[row] = 2 * ep + (pivot ? 1 : 0);
#pragma unroll
      for (int t = 0; t < CPT; ++t) U[(half * CPT + t) * ROWS + row] = fx::split(pv[t], tk[t], ep);
    }
    if (other) {
      int e = fx::kNone;
      double x[BW];  // read again rather than held over the barrier: at 100 rows 122 registers, not 174
#pragma unroll
      for (int k = 0; k < BW; ++k) {
        x[k] = k < kb ? M[rows[k] * LD + tid] : 0.0;
        e = max(e, fx::exponent_of(x[k], -ts[k]));
      }
      eX[tid] = e;
#pragma unroll
      for (int k = 0; k < BW; ++k) X[k * COLS + tid] = fx::split(x[k], -ts[k], e);
    }
    __syncthreads();
    // ---- M[:, j] = (M[:, j] or 0) + U x_P[:, j], tiles of 4 rows x 2 columns per thread ----
    constexpr int TJ = COLS / 2, TI = ROWS / 4;
    const bool first = kb == NB;
    for (int tile = tid; tile < TI * TJ && !first; tile += THREADS) {
      const int j = tile % TJ * 2, i = tile / TJ * 4;
      if (j >= c0 && j + 1 < c0 + kb) continue;  // the panel's own columns
      fx::Acc a[4][2];
#pragma unroll
      for (int k = 0; k < BW; ++k) {
        const int4 u01 = *reinterpret_cast<const int4*>(U + k * ROWS + i);
        const int4 u23 = *reinterpret_cast<const int4*>(U + k * ROWS + i + 2);
        const int4 x01 = *reinterpret_cast<const int4*>(X + k * COLS + j);
        const int2 u[4] = {make_int2(u01.x, u01.y), make_int2(u01.z, u01.w), make_int2(u23.x, u23.y),
                           make_int2(u23.z, u23.w)};
        const int2 x[2] = {make_int2(x01.x, x01.y), make_int2(x01.z, x01.w)};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 2; ++q) fx::mad(a[p][q], u[p], x[q]);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int jj = j + q;
        if (jj >= NB || (jj >= c0 && jj < c0 + kb)) continue;
#pragma unroll
        for (int p = 0; p < 4; ++p)
          if (i + p < NB) {
            double* m = M + (i + p) * LD + jj;
            const int eu = eU[i + p];  // exponent times two, and in bit 0 whether the row is a pivot row
            *m = fma(fx::value(a[p][q]), fx::scale(eu >> 1, eX[jj]), eu & 1 ? 0.0 : *m);
          }
      }
    }
    __syncthreads();
  }
}

}  // namespace gjfx
}  // namespace frk
