// FR/CPR residual R(U) and the finite-difference operator A z of Sec. 3 / 4.5.
//
// One thread per (element, solution point); EPB = 256 / Np elements per CTA.
// Per element, in shared memory: the (possibly perturbed) state, the
// transformed fluxes F = (hy/2) f, G = (hx/2) g at the solution points, and
// the common fluxes F^num on the 4 (p+1) face points.  Fluxes are kept in
// physical form (f, g, f_n); the metric factors |J| |grad xi| / |J| = 2/hx,
// 2/hy are applied once per output.  A face point's own
// trace comes from shared memory, the neighbour's from global memory (L2),
// both summed in the same order with the same coefficients, so the two
// elements sharing a face compute bit-identical common fluxes (discrete
// conservation holds to round-off).  The corrected divergence uses the
// folded derivative matrix Dt (the local-flux traces F^l(+-1) are absorbed
// into Dt, which removes their extrapolation from the flop count).
//
// Bound: FP64 issue (two operations per clock and SM).  At 512^2, p = 3, R and
// A z with its two norms take 2114 us together; with IEEE divisions, roots and
// fmax in the fluxes, two divisions per thread for the metric and one load in
// flight in the norms they took 2718 us.
#include "residual_body.cuh"

namespace frk {
namespace {

template <int P, int MODE, int TV, int RM>
__global__ void __launch_bounds__(TV == 2 ? 128 : 256, 4) k_residual(const __grid_constant__ ResArgs a) {
  __shared__ ResSmem<P, TV> sm;
  if (a.done && *a.done) return;
  residual_body<P, MODE, TV, RM>(a, a.z, a.b, a.eps2, a.out, blockIdx.x, sm);
}

// A z of Arnoldi iteration j of every instance (of one degree) in one grid:
// instance k owns the tiles [start[k], start[k+1]); its table entry holds
// the basis in `out`, and A z is written to V_{j+1}.
template <int P, int RM>
__global__ void __launch_bounds__(256, 4) kb_residual(const ResArgs* __restrict__ tab, const int* __restrict__ start,
                                                      int ninst, int j) {
  const int k = batch_instance(start, ninst, blockIdx.x);
  const ResArgs& a = tab[k];
  const long long ndof = a.ne * 4 * (P + 1) * (P + 1);
  __shared__ ResSmem<P, 0> sm;
  if (*a.done) return;
  residual_body<P, 1, 0, RM>(a, a.z, nullptr, a.eps2, a.out + (size_t)(j + 1) * ndof, blockIdx.x - start[k], sm);
}

// A z with FP32 linear parts (jv_precision 1).  R(U+eps z) - R(U) is the
// corrected divergence of the flux differences dF = F(U+eps z) - F(U) at the
// points and df = f^num(U+eps z) - f^num(U) on the faces; the divergence and
// correction are linear, so they run in FP32 on dF, df.  The nonlinear parts
// stay FP64: the pointwise fluxes at U + eps z and their difference from the
// cached F(U), the face states q(U) + eps trace(z) (trace of z in FP32, the
// state itself in FP64) and the Rusanov fluxes at them, differenced against
// the cached f^num(U).  Same element tiles as k_residual; MODE 1: A z,
// MODE 2: b - A z.
template <int P, int MODE, int TV, int RM>
__global__ void __launch_bounds__(256) k_jv32(const ResArgs a) {
  constexpr int N = P + 1, NP = N * N;
  constexpr int TX = Tile<P, TV>::TX, TY = Tile<P, TV>::TY, NE = TX * TY;
  constexpr int NXF = (TX + 1) * TY * N;
  constexpr int NYF = (TY + 1) * TX * N;
  __shared__ float sdF[NE][4][NP], sdG[NE][4][NP], sz[NE][4][NP];
  __shared__ float strz[NE][4][4][N];         // own traces of z [face W,E,S,N][var][k]
  __shared__ float shzx[2][TY][4][N];         // outside traces of z on the tile's west / east faces
  __shared__ float shzy[2][TX][4][N];         // outside traces of z on the tile's south / north faces
  constexpr int NOWN = NE * 4 * N, NHALO = 2 * (TX + TY) * N;
  __shared__ float sfx[TY][TX + 1][4][N];     // df on x-faces
  __shared__ float sfy[TX][TY + 1][4][N];     // df on y-faces
  __shared__ float sDt[N][N], slm[N], slp[N], sdgL[N], sdgR[N];

  if (a.done && *a.done) return;
  if (threadIdx.x < N * N) sDt[threadIdx.x / N][threadIdx.x % N] = (float)a.tab.Dt[threadIdx.x / N][threadIdx.x % N];
  if (threadIdx.x < N) {
    slm[threadIdx.x] = (float)a.tab.lm[threadIdx.x];
    slp[threadIdx.x] = (float)a.tab.lp[threadIdx.x];
    sdgL[threadIdx.x] = (float)a.tab.dgL[threadIdx.x];
    sdgR[threadIdx.x] = (float)a.tab.dgR[threadIdx.x];
  }
  const int tiles_x = (a.nx + TX - 1) / TX;
  const int ix0 = (int)(blockIdx.x % tiles_x) * TX, iy0 = (int)(blockIdx.x / tiles_x) * TY;
  const int ax = min(TX, a.nx - ix0), ay = min(TY, a.ny - iy0);
  const int el = threadIdx.x / NP, t = threadIdx.x % NP;
  const int lx = el % TX, ly = el / TX;
  const bool active = el < NE && lx < ax && ly < ay;
  const long long e = (long long)(ix0 + lx) + (long long)a.nx * (iy0 + ly);
  const double eps = a.eps2[0], ieps = a.eps2[1];
  // ---- 1: perturbed state, point fluxes (FP64) and their differences ----
  if (active) {
    const long long base = e * 4 * NP + t;
    double q[4], f[4], g[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long o = base + v * NP;
      const double zv = a.z[o];
      q[v] = fma(eps, zv, a.U[o]);
      sz[el][v][t] = (float)zv;
    }
    euler_fluxes(q, a.gam, f, g);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      sdF[el][v][t] = (float)(f[v] - a.lin_fg[(e * 8 + v) * NP + t]);
      sdG[el][v][t] = (float)(g[v] - a.lin_fg[(e * 8 + 4 + v) * NP + t]);
    }
  }
  __syncthreads();
  // ---- 2a: own traces of z (FP32), then the outside neighbours' traces of z
  //      on the tile's boundary faces (separate work items, from global memory) ----
  for (int idx = threadIdx.x; idx < NOWN + NHALO; idx += blockDim.x) {
    if (idx < NOWN) {
      const int e2 = idx / (4 * N), face = (idx / N) % 4, k = idx % N;
      if ((e2 % TX) >= ax || (e2 / TX) >= ay) continue;
      const int off = face < 2 ? N * k : k;
      const int stride = face < 2 ? 1 : N;
      const float* c = (face == 0 || face == 2) ? slm : slp;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float s2 = c[0] * sz[e2][v][off];
#pragma unroll
        for (int q = 1; q < N; ++q) s2 = fmaf(c[q], sz[e2][v][off + q * stride], s2);
        strz[e2][face][v][k] = s2;
      }
    } else {
      const int h = idx - NOWN, seg = h / N, k = h % N;
      long long nb;
      int off, stride;
      const double* c;
      float* dst;
      if (seg < 2 * TY) {
        const int side = seg / TY, fy = seg % TY;
        if (fy >= ay) continue;
        const int gx = side == 0 ? (ix0 + a.nx - 1) % a.nx : (ix0 + ax) % a.nx;
        nb = (long long)gx + (long long)a.nx * (iy0 + fy);
        off = N * k;
        stride = 1;
        c = side == 0 ? a.tab.lp : a.tab.lm;
        dst = &shzx[side][fy][0][k];
      } else {
        const int s2 = seg - 2 * TY, side = s2 / TX, fx = s2 % TX;
        if (fx >= ax) continue;
        const int gy = side == 0 ? (iy0 + a.ny - 1) % a.ny : (iy0 + ay) % a.ny;
        nb = (long long)(ix0 + fx) + (long long)a.nx * gy;
        off = k;
        stride = N;
        c = side == 0 ? a.tab.lp : a.tab.lm;
        dst = &shzy[side][fx][0][k];
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) dst[v * N] = (float)trace_sum<N>(a.z + nb * 4 * NP + v * NP + off, stride, c);
    }
  }
  __syncthreads();
  // ---- 2b: face states q(U) + eps trace(z), Rusanov (FP64), df ----
  for (int idx = threadIdx.x; idx < NXF + NYF; idx += blockDim.x) {
    double qm[4], qp[4], fc[4];
    float tzm[4], tzp[4];
    const double* cache;
    int dir;
    int sx0, sx1, sx2, sx3;  // destination (row/column, face index, -, k)
    if (idx < NXF) {
      const int k = idx % N, rr = idx / N, xf = rr % (TX + 1), fy = rr / (TX + 1);
      if (fy >= ay || xf > ax) continue;
      const int gy = iy0 + fy;
      const long long ep = (long long)((ix0 + xf) % a.nx) + (long long)a.nx * gy;  // element east of the face
      cache = a.lin_fx + (ep * N + k) * 12;
      const float* pm = xf >= 1 ? &strz[xf - 1 + TX * fy][1][0][k] : &shzx[0][fy][0][k];
      const float* pp = xf < ax ? &strz[xf + TX * fy][0][0][k] : &shzx[1][fy][0][k];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        tzm[v] = pm[v * N];
        tzp[v] = pp[v * N];
      }
      dir = 0; sx0 = fy; sx1 = xf; sx3 = k; sx2 = 0;
    } else {
      const int i2 = idx - NXF;
      const int k = i2 % N, rr = i2 / N, yf = rr % (TY + 1), fx = rr / (TY + 1);
      if (fx >= ax || yf > ay) continue;
      const int gx = ix0 + fx;
      const long long ep = (long long)gx + (long long)a.nx * ((iy0 + yf) % a.ny);  // element north of the face
      cache = a.lin_fy + (ep * N + k) * 12;
      const float* pm = yf >= 1 ? &strz[fx + TX * (yf - 1)][3][0][k] : &shzy[0][fx][0][k];
      const float* pp = yf < ay ? &strz[fx + TX * yf][2][0][k] : &shzy[1][fx][0][k];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        tzm[v] = pm[v * N];
        tzp[v] = pp[v * N];
      }
      dir = 1; sx0 = fx; sx1 = yf; sx3 = k; sx2 = 0;
    }
    (void)sx2;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      qm[v] = fma(eps, (double)tzm[v], cache[v]);
      qp[v] = fma(eps, (double)tzp[v], cache[4 + v]);
    }
    riemann_flux(RM, qm, qp, dir, a.gam, fc);
    if (dir == 0) {
#pragma unroll
      for (int v = 0; v < 4; ++v) sfx[sx0][sx1][v][sx3] = (float)(fc[v] - cache[8 + v]);
    } else {
#pragma unroll
      for (int v = 0; v < 4; ++v) sfy[sx0][sx1][v][sx3] = (float)(fc[v] - cache[8 + v]);
    }
  }
  __syncthreads();
  // ---- 3: corrected divergence of the differences (FP32), output (FP64) ----
  if (!active) return;
  const float sx = (float)a.sx[ix0 + lx], sy = (float)a.sy[iy0 + ly];
  const int i = t % N, j = t / N;
  const long long base = e * 4 * NP + t;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    float dF = sdgL[i] * sfx[ly][lx][v][j];
    dF = fmaf(sdgR[i], sfx[ly][lx + 1][v][j], dF);
#pragma unroll
    for (int k = 0; k < N; ++k) dF = fmaf(sDt[i][k], sdF[el][v][k + N * j], dF);
    float dG = sdgL[j] * sfy[lx][ly][v][i];
    dG = fmaf(sdgR[j], sfy[lx][ly + 1][v][i], dG);
#pragma unroll
    for (int k = 0; k < N; ++k) dG = fmaf(sDt[j][k], sdG[el][v][i + N * k], dG);
    const float dR = -fmaf(sx, dF, sy * dG);  // R(U + eps z) - R(U)
    const long long o = base + v * NP;
    const double zo = a.z[o];
    const double Az = eps > 0.0 ? fma(-(double)dR, ieps, a.shift * zo) : a.shift * zo;
    a.out[o] = MODE == 2 ? a.b[o] - Az : Az;
  }
}

template <int P, int TV, int RM>
int launch_pvr(fr_ctx* ctx, int mode, const ResArgs& a, cudaStream_t s) {
  constexpr int NP = (P + 1) * (P + 1), TX = Tile<P, TV>::TX, TY = Tile<P, TV>::TY;
  const long long grid = (long long)((ctx->nx + TX - 1) / TX) * ((ctx->ny + TY - 1) / TY);
  const dim3 blk(TX * TY * NP);
  // algorithmic work: R reads U and writes R (16 B/DOF); A z also reads z and
  // R0 (and b) and adds the perturbation and the difference quotient.  Inside
  // a GMRES cycle the work is booked per finished iteration instead.
  const double nd = (double)ctx->ndof, fl = residual_flops_per_element(P) * (double)ctx->ne;
  const bool in_cycle = a.done != nullptr;
  const double wb = in_cycle ? 0.0 : (mode == 0 ? 16.0 : (mode == 1 ? 32.0 : 40.0)) * nd;
  const double wf = in_cycle ? 0.0 : (mode == 0 ? fl : fl + 6.0 * nd);
  const bool mixed = ctx->opts.jv_precision == 1;
  if constexpr (TV != 2) {
    if (mode == 3) { ProfScope ps_(ctx, FR_KF_OTHER, s); k_residual<P, 3, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
    else if (mode == 1 && mixed) { ProfScope ps_(ctx, FR_KF_JV, s, wb, wf); k_jv32<P, 1, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
    else if (mode == 2 && mixed) { ProfScope ps_(ctx, FR_KF_JV, s, wb, wf); k_jv32<P, 2, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
  }
  if (mode == 0) { ProfScope ps_(ctx, FR_KF_RESIDUAL, s, wb, wf); k_residual<P, 0, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
  else if (mode == 1 && !mixed) { ProfScope ps_(ctx, FR_KF_JV, s, wb, wf); k_residual<P, 1, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
  else if (mode == 2 && !mixed) { ProfScope ps_(ctx, FR_KF_JV, s, wb, wf); k_residual<P, 2, TV, RM><<<(unsigned)grid, blk, 0, s>>>(a); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

// Shape-0 tiles of 9 to 25 elements keep a CTA busy for 20 us, so a mesh with
// fewer of them than the chip has SMs runs on a fraction of its FP64 units; the
// small tiles repeat more halo traces (about a third more FP64 work) but spread.
template <int P>
bool use_small_tile(const fr_ctx* ctx, int mode) {
  if (ctx->tile_variant != 0 || mode == 3 || (mode != 0 && ctx->opts.jv_precision == 1)) return false;
  constexpr int TX = Tile<P, 0>::TX, TY = Tile<P, 0>::TY;
  const long long tiles = (long long)((ctx->nx + TX - 1) / TX) * ((ctx->ny + TY - 1) / TY);
  return tiles < ctx->num_sms;
}

// the common flux is a template parameter so each flux gets its own register allocation
template <int P, int TV>
int launch_pv(fr_ctx* ctx, int mode, const ResArgs& a, cudaStream_t s) {
  return a.riemann == 1 ? launch_pvr<P, TV, 1>(ctx, mode, a, s) : launch_pvr<P, TV, 0>(ctx, mode, a, s);
}

template <int P>
int launch_p(fr_ctx* ctx, int mode, const ResArgs& a, cudaStream_t s) {
  if (use_small_tile<P>(ctx, mode)) return launch_pv<P, 2>(ctx, mode, a, s);
  return ctx->tile_variant == 1 ? launch_pv<P, 1>(ctx, mode, a, s) : launch_pv<P, 0>(ctx, mode, a, s);
}

}  // namespace

ResArgs residual_args(fr_ctx* ctx, const double* U, const double* R0, double shift) {
  ResArgs a{};
  a.U = U; a.R0 = R0;
  a.sx = ctx->sx; a.sy = ctx->sy;
  a.ne = ctx->ne; a.nx = ctx->nx; a.ny = ctx->ny;
  a.gam = ctx->opts.gamma; a.shift = shift;
  a.eps_rel = ctx->opts.eps_rel; a.eps_fixed = ctx->opts.eps_fixed;
  a.lin_fg = ctx->lin_fg; a.lin_fx = ctx->lin_fx; a.lin_fy = ctx->lin_fy;
  a.riemann = ctx->opts.riemann;
  a.tab = ctx->tab;
  return a;
}

bool residual_small_tile(const fr_ctx* ctx) {
  switch (ctx->p) {
    case 2: return use_small_tile<2>(ctx, 1);
    case 3: return use_small_tile<3>(ctx, 1);
    case 4: return use_small_tile<4>(ctx, 1);
    default: return false;
  }
}

int launch_residual(fr_ctx* ctx, int mode, const double* U, const double* z, const double* R0,
                    const double* b, double* out, double shift, const double* eps2,
                    const int* done, cudaStream_t s) {
  if (ctx->dim3) return launch_f3_residual(ctx, mode, U, z, R0, b, out, shift, eps2, done, s);
  if (ctx->viscous) return launch_ns_residual(ctx, mode, U, z, R0, b, out, shift, eps2, done, s);
  ResArgs a = residual_args(ctx, U, R0, shift);
  a.z = z; a.b = b; a.out = out; a.eps2 = eps2; a.done = done;
  switch (ctx->p) {
    case 2: return launch_p<2>(ctx, mode, a, s);
    case 3: return launch_p<3>(ctx, mode, a, s);
    case 4: return launch_p<4>(ctx, mode, a, s);
    case 5: return launch_p<5>(ctx, mode, a, s);
    case 6: return launch_p<6>(ctx, mode, a, s);
    default: return set_error(ctx, FR_ERR_UNSUPPORTED, "degree %d not compiled", ctx->p);
  }
}

size_t batch_residual_bytes() { return sizeof(ResArgs); }

// tiles of the residual launch (tile variant 0, the one the batched launch uses)
unsigned residual_grid_of(const fr_ctx* ctx) {
  int tx = 1, ty = 1;
  switch (ctx->p) {
    case 2: tx = Tile<2, 0>::TX; ty = Tile<2, 0>::TY; break;
    case 3: tx = Tile<3, 0>::TX; ty = Tile<3, 0>::TY; break;
    case 4: tx = Tile<4, 0>::TX; ty = Tile<4, 0>::TY; break;
    default: return 0;
  }
  return (unsigned)(((ctx->nx + tx - 1) / tx) * ((ctx->ny + ty - 1) / ty));
}

// table entry of the batched A z: A = shift I - dR/dU at U, z = the
// context's preconditioned vector, output base = the Krylov basis
int fill_batch_residual(fr_ctx* ctx, const double* U, const double* R0, double shift, void* out) {
  if (ctx->dim3 || ctx->viscous || ctx->opts.jv_precision != 0 || ctx->p < 2 || ctx->p > 4) return FR_ERR_UNSUPPORTED;
  ResArgs a = residual_args(ctx, U, R0, shift);
  a.z = ctx->z; a.out = ctx->V;
  a.eps2 = ctx->scal + S_EPS; a.done = ctx->gd.done;
  *reinterpret_cast<ResArgs*>(out) = a;
  return FR_OK;
}

int launch_batch_residual(int p, int riemann, const void* tab, const int* start, int ninst, int nblocks, int j,
                          cudaStream_t s) {
  const ResArgs* t = reinterpret_cast<const ResArgs*>(tab);
  count_launch();
  switch (p) {
    case 2: riemann ? kb_residual<2, 1><<<nblocks, Tile<2, 0>::TX * Tile<2, 0>::TY * 9, 0, s>>>(t, start, ninst, j)
                    : kb_residual<2, 0><<<nblocks, Tile<2, 0>::TX * Tile<2, 0>::TY * 9, 0, s>>>(t, start, ninst, j); break;
    case 3: riemann ? kb_residual<3, 1><<<nblocks, Tile<3, 0>::TX * Tile<3, 0>::TY * 16, 0, s>>>(t, start, ninst, j)
                    : kb_residual<3, 0><<<nblocks, Tile<3, 0>::TX * Tile<3, 0>::TY * 16, 0, s>>>(t, start, ninst, j); break;
    case 4: riemann ? kb_residual<4, 1><<<nblocks, Tile<4, 0>::TX * Tile<4, 0>::TY * 25, 0, s>>>(t, start, ninst, j)
                    : kb_residual<4, 0><<<nblocks, Tile<4, 0>::TX * Tile<4, 0>::TY * 25, 0, s>>>(t, start, ninst, j); break;
    default: return FR_ERR_UNSUPPORTED;
  }
  return cudaGetLastError() == cudaSuccess ? FR_OK : FR_ERR_CUDA;
}

int launch_linearize(fr_ctx* ctx, const double* U, cudaStream_t s) {
  if (ctx->dim3) return launch_f3_linearize(ctx, U, s);
  if (ctx->opts.jv_precision != 1 || ctx->viscous) return FR_OK;
  return launch_residual(ctx, 3, U, nullptr, nullptr, nullptr, nullptr, 0.0, nullptr, nullptr, s);
}

}  // namespace frk
