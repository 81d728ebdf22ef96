// The tile of the Euler FR residual and of its finite-difference products, shared
// by the per-product kernels (residual.cu) and the GMRES cycle kernel (cycle.cuh).
// No pointer here is restrict-qualified: in the cycle kernel z is written by other
// CTAs of the same launch, so its loads must not take the read-only path.
#pragma once

#include "device.cuh"

namespace frk {

struct ResArgs {
  const double* U;
  const double* z;
  const double* R0;
  const double* b;
  double* out;
  const double* sx;    // 2 / hx per element column
  const double* sy;    // 2 / hy per element row
  const double* eps2;  // (eps, 1/eps) of the FD product
  const int* done;
  long long ne;
  int nx, ny;
  double gam;
  double shift;
  double eps_rel;
  double eps_fixed;
  double* lin_fg;  // mode 3 writes / mixed A z reads: F(U), G(U) [ne][8][NP]
  double* lin_fx;  // per element's west face point: q-, q+, f^num (4 each) [ne][N][12]
  double* lin_fy;  // per element's south face point, same layout
  int riemann;     // common flux: 0 Rusanov, 1 Roe
  Tables tab;
};

// sum_k c[k] * x[k*stride], fixed order, explicit FMAs
template <int N>
__device__ __forceinline__ double trace_sum(const double* x, int stride,
                                            const double* c) {
  double s = c[0] * x[0];
#pragma unroll
  for (int k = 1; k < N; ++k) s = fma(c[k], x[k * stride], s);
  return s;
}

// neighbour trace from global memory, optionally perturbed by eps * z
template <int N, bool PERTURB>
__device__ __forceinline__ double trace_global(const double* U, const double* z, long long off,
                                               int stride, const double* c, double eps) {
  if (!PERTURB) return trace_sum<N>(U + off, stride, c);
  double s = c[0] * fma(eps, z[off], U[off]);
#pragma unroll
  for (int k = 1; k < N; ++k) s = fma(c[k], fma(eps, z[off + k * stride], U[off + k * stride]), s);
  return s;
}

// Element tile handled by one CTA (TX x TY elements, one thread per point);
// two shapes per degree, picked at run time by the autotuner.
template <int P, int V> struct Tile;
template <> struct Tile<2, 0> { static constexpr int TX = 5, TY = 5; };
template <> struct Tile<2, 1> { static constexpr int TX = 7, TY = 4; };
template <> struct Tile<3, 0> { static constexpr int TX = 4, TY = 4; };
template <> struct Tile<3, 1> { static constexpr int TX = 8, TY = 2; };
template <> struct Tile<4, 0> { static constexpr int TX = 3, TY = 3; };
template <> struct Tile<4, 1> { static constexpr int TX = 5, TY = 2; };
template <> struct Tile<5, 0> { static constexpr int TX = 2, TY = 3; };
template <> struct Tile<5, 1> { static constexpr int TX = 3, TY = 2; };
template <> struct Tile<6, 0> { static constexpr int TX = 2, TY = 2; };
template <> struct Tile<6, 1> { static constexpr int TX = 5, TY = 1; };
// Shape 2: small meshes, whose shape-0 tiles would leave most SMs idle (see use_small_tile).
template <> struct Tile<2, 2> { static constexpr int TX = 2, TY = 2; };
template <> struct Tile<3, 2> { static constexpr int TX = 2, TY = 2; };
template <> struct Tile<4, 2> { static constexpr int TX = 2, TY = 1; };
template <> struct Tile<5, 2> { static constexpr int TX = 2, TY = 1; };
template <> struct Tile<6, 2> { static constexpr int TX = 1, TY = 1; };

// Shared memory of one tile.
template <int P, int TV> struct ResSmem {
  static constexpr int N = P + 1, NP = N * N, TX = Tile<P, TV>::TX, TY = Tile<P, TV>::TY, NE = TX * TY;
  double sq[NE][4][NP];
  double sF[NE][4][NP];
  double sG[NE][4][NP];
  double str[NE][4][4][N];       // own traces [face W,E,S,N][var][k]
  double shx[2][TY][4][N];       // outside traces on the tile's west / east faces
  double shy[2][TX][4][N];       // outside traces on the tile's south / north faces
  double sfx[TY][TX + 1][4][N];  // common flux f_n on x-face xf of tile row ly
  double sfy[TX][TY + 1][4][N];  // common flux g_n on y-face yf of tile column lx
  double sDt[N][N], slm[N], slp[N], sdgL[N], sdgR[N];
};

// One tile of R(U) (MODE 0), A z (1) or b - A z (2; 4: b - A z, or A z where b is
// null); eps2: (eps, 1/eps) of the product.
template <int P, int MODE, int TV, int RM>
__device__ __forceinline__ void residual_body(const ResArgs& a, const double* z, const double* b, const double* eps2,
                                              double* out, int bid, ResSmem<P, TV>& sm) {
  constexpr int N = P + 1, NP = N * N;
  constexpr int TX = Tile<P, TV>::TX, TY = Tile<P, TV>::TY, NE = TX * TY;
  constexpr int NXF = (TX + 1) * TY * N;  // points on the tile's x-faces (normal +x)
  constexpr int NYF = (TY + 1) * TX * N;  // points on the tile's y-faces (normal +y)
  constexpr bool PERTURB = MODE == 1 || MODE == 2 || MODE == 4;  // MODE 3: R's fluxes at U into the caches
  // MODE 3 feeds the FP32-linear-parts product, which repeats its fluxes with
  // the correctly rounded operations; the others take the fast ones, whose
  // common flux comes out doubled (sdgL, sdgR carry the 1/2)
  constexpr bool FAST = MODE != 3;
  auto& sq = sm.sq; auto& sF = sm.sF; auto& sG = sm.sG; auto& str = sm.str;
  auto& shx = sm.shx; auto& shy = sm.shy; auto& sfx = sm.sfx; auto& sfy = sm.sfy;
  auto& sDt = sm.sDt; auto& slm = sm.slm; auto& slp = sm.slp; auto& sdgL = sm.sdgL; auto& sdgR = sm.sdgR;
  constexpr int NOWN = NE * 4 * N;           // own-trace work items
  constexpr int NHALO = 2 * (TX + TY) * N;   // outside-trace work items

  if (threadIdx.x < N * N) sDt[threadIdx.x / N][threadIdx.x % N] = a.tab.Dt[threadIdx.x / N][threadIdx.x % N];
  if (threadIdx.x < N) {
    slm[threadIdx.x] = a.tab.lm[threadIdx.x];
    slp[threadIdx.x] = a.tab.lp[threadIdx.x];
    sdgL[threadIdx.x] = 0.5 * a.tab.dgL[threadIdx.x];
    sdgR[threadIdx.x] = 0.5 * a.tab.dgR[threadIdx.x];
  }

  const int tiles_x = (a.nx + TX - 1) / TX;
  const int ix0 = (int)(bid % tiles_x) * TX, iy0 = (int)(bid / tiles_x) * TY;
  const int ax = min(TX, a.nx - ix0), ay = min(TY, a.ny - iy0);  // active tile extent
  const int el = threadIdx.x / NP, t = threadIdx.x % NP;
  const int lx = el % TX, ly = el / TX;
  const bool active = el < NE && lx < ax && ly < ay;  // blockDim >= NE * NP
  const long long e = (long long)(ix0 + lx) + (long long)a.nx * (iy0 + ly);

  double eps = 0.0, ieps = 0.0;
  if (PERTURB) {
    eps = eps2[0];
    ieps = eps2[1];
  }
  // on small tiles, which wait for latency and have registers to spare, the
  // metric and the output's other operands are loaded with the state
  constexpr bool EARLY = TV == 2;
  double sx = 0.0, sy = 0.0, zo[4], r0[4];
  // ---- 1: state (perturbed for A z) and pointwise fluxes ----
  if (active) {
    double q[4], f[4], g[4];
    const long long base = e * 4 * NP + t;
    if (EARLY) {
      sx = a.sx[ix0 + lx];
      sy = a.sy[iy0 + ly];
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long o = base + v * NP;
      if (EARLY && PERTURB) {
        zo[v] = z[o];
        r0[v] = a.R0[o];
        q[v] = fma(eps, zo[v], a.U[o]);
      } else {
        q[v] = PERTURB ? fma(eps, z[o], a.U[o]) : a.U[o];
      }
      sq[el][v][t] = q[v];
    }
    euler_fluxes<FAST>(q, a.gam, f, g);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      sF[el][v][t] = f[v];
      sG[el][v][t] = g[v];
      if (MODE == 3) {
        a.lin_fg[(e * 8 + v) * NP + t] = f[v];
        a.lin_fg[(e * 8 + 4 + v) * NP + t] = g[v];
      }
    }
  }
  // the outside neighbours' traces on the tile's boundary faces, from global
  // memory: before the barrier, so their latency is the state's too, and from the
  // last threads, which small tiles leave free
  for (int h = (int)blockDim.x - 1 - (int)threadIdx.x; h < NHALO; h += blockDim.x) {
    const int seg = h / N, k = h % N;
    long long nb;
    int off, stride;
    double* dst;
    int side;
    if (seg < 2 * TY) {  // west (side 0) / east (side 1) boundary of tile row fy
      side = seg / TY;
      const int fy = seg % TY;
      if (fy >= ay) continue;
      const int gx = side == 0 ? (ix0 + a.nx - 1) % a.nx : (ix0 + ax) % a.nx;
      nb = (long long)gx + (long long)a.nx * (iy0 + fy);
      off = N * k;
      stride = 1;
      dst = &shx[side][fy][0][k];
    } else {             // south (side 0) / north (side 1) boundary of tile column fx
      const int s2 = seg - 2 * TY, fx = s2 % TX;
      side = s2 / TX;
      if (fx >= ax) continue;
      const int gy = side == 0 ? (iy0 + a.ny - 1) % a.ny : (iy0 + ay) % a.ny;
      nb = (long long)(ix0 + fx) + (long long)a.nx * gy;
      off = k;
      stride = N;
      dst = &shy[side][fx][0][k];
    }
    double c[N];  // the west neighbour's east trace, the east one's west trace, ...
#pragma unroll
    for (int l = 0; l < N; ++l) c[l] = side == 0 ? a.tab.lp[l] : a.tab.lm[l];
#pragma unroll
    for (int v = 0; v < 4; ++v)
      dst[v * N] = trace_global<N, PERTURB>(a.U, z, nb * 4 * NP + v * NP + off, stride, c, eps);
  }
  __syncthreads();
  // ---- 2a: own solution traces on the four faces of every tile element ----
  for (int idx = threadIdx.x; idx < NOWN; idx += blockDim.x) {
    const int e2 = idx / (4 * N), face = (idx / N) % 4, k = idx % N;
    if ((e2 % TX) >= ax || (e2 / TX) >= ay) continue;
    const int off = face < 2 ? N * k : k;
    const int stride = face < 2 ? 1 : N;
    const double* c = (face == 0 || face == 2) ? slm : slp;
#pragma unroll
    for (int v = 0; v < 4; ++v) str[e2][face][v][k] = trace_sum<N>(&sq[e2][v][off], stride, c);
  }
  __syncthreads();
  // ---- 2b: one common flux per face point, both traces from shared memory; one
  //      flux for both directions, so a warp that holds faces of both runs it once ----
  for (int idx = threadIdx.x; idx < NXF + NYF; idx += blockDim.x) {
    const double *pm, *pp;
    double *dst, *cache = nullptr;
    int dir;
    if (idx < NXF) {
      const int k = idx % N, rr = idx / N, xf = rr % (TX + 1), fy = rr / (TX + 1);
      if (fy >= ay || xf > ax) continue;
      pm = xf >= 1 ? &str[xf - 1 + TX * fy][1][0][k] : &shx[0][fy][0][k];
      pp = xf < ax ? &str[xf + TX * fy][0][0][k] : &shx[1][fy][0][k];
      dst = &sfx[fy][xf][0][k];
      dir = 0;
      if (MODE == 3 && xf < ax)  // the west face of tile element xf
        cache = a.lin_fx + (((long long)(ix0 + xf) + (long long)a.nx * (iy0 + fy)) * N + k) * 12;
    } else {
      const int i2 = idx - NXF;
      const int k = i2 % N, rr = i2 / N, yf = rr % (TY + 1), fx = rr / (TY + 1);
      if (fx >= ax || yf > ay) continue;
      pm = yf >= 1 ? &str[fx + TX * (yf - 1)][3][0][k] : &shy[0][fx][0][k];
      pp = yf < ay ? &str[fx + TX * yf][2][0][k] : &shy[1][fx][0][k];
      dst = &sfy[fx][yf][0][k];
      dir = 1;
      if (MODE == 3 && yf < ay)  // the south face of tile element yf
        cache = a.lin_fy + (((long long)(ix0 + fx) + (long long)a.nx * (iy0 + yf)) * N + k) * 12;
    }
    double qm[4], qp[4], fc[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      qm[v] = pm[v * N];
      qp[v] = pp[v * N];
    }
    // the caches' flux is subtracted from one at U + eps z and the difference divided by
    // eps, which shows its last bits: it keeps one expression per direction, as those
    // bits depend on how the compiler contracts it
    if (FAST) riemann_flux2(RM, qm, qp, dir, a.gam, fc);
    else if (dir == 0) riemann_flux(RM, qm, qp, 0, a.gam, fc);
    else riemann_flux(RM, qm, qp, 1, a.gam, fc);
#pragma unroll
    for (int v = 0; v < 4; ++v) dst[v * N] = fc[v];
    if (MODE == 3 && cache) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        cache[v] = qm[v];
        cache[4 + v] = qp[v];
        cache[8 + v] = fc[v];
      }
    }
  }
  __syncthreads();

  // ---- 3: corrected divergence and the output ----
  if (MODE == 3 || !active) return;
  const int i = t % N, j = t / N;
  // with unscaled fluxes, -(1/|J|)(dF~/dxi + dG~/deta) = -(2/hx) df~ - (2/hy) dg~
  if (!EARLY) {
    sx = a.sx[ix0 + lx];
    sy = a.sy[iy0 + ly];
  }
  const long long base = e * 4 * NP + t;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    double dF = sdgL[i] * sfx[ly][lx][v][j];
    dF = fma(sdgR[i], sfx[ly][lx + 1][v][j], dF);
#pragma unroll
    for (int k = 0; k < N; ++k) dF = fma(sDt[i][k], sF[el][v][k + N * j], dF);
    double dG = sdgL[j] * sfy[lx][ly][v][i];
    dG = fma(sdgR[j], sfy[lx][ly + 1][v][i], dG);
#pragma unroll
    for (int k = 0; k < N; ++k) dG = fma(sDt[j][k], sG[el][v][i + N * k], dG);
    const double R = -fma(sx, dF, sy * dG);
    const long long o = base + v * NP;
    if (MODE == 0) {
      out[o] = R;
    } else {
      const double zv = EARLY ? zo[v] : z[o], rv = EARLY ? r0[v] : a.R0[o];
      const double Az = eps > 0.0 ? fma(-(R - rv), ieps, a.shift * zv) : a.shift * zv;
      out[o] = MODE == 2 || (MODE == 4 && b) ? b[o] - Az : Az;
    }
  }
}

}  // namespace frk
