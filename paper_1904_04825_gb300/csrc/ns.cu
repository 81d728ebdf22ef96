// Viscous (Navier-Stokes) FR residual with BR2 common gradients, Sec. 2-3
// (Eqs. com_q, com_grad_q and the BR2 lifting with g'(+-1) = +-(P+1)(P+2)/2).
//
// R(U), A z and b - A z take three kernels, FP64-issue bound:
//  k_ns_trace: per element, the (possibly perturbed) state q and its normal
//    derivative traced to the 4 (p+1) face points -> trace buffer.  The
//    tangential derivative is not traced: it is the derivative along the face
//    of the common solution, which k_ns_face takes once for both elements.
//  k_ns_face:  per west / south face point (and north wall), the common
//    solution, the BR2 common gradient and the common total flux (Rusanov
//    inviscid minus viscous) -> face buffer, each face once.
//  k_ns_cell:  per element, the FR-corrected gradient and total flux at the
//    solution points, the corrected divergence with the four faces' common
//    fluxes, the body-force source and the output.  Both elements of a face
//    read the same stored flux, so conservation holds to round-off.
// Bound: FP64 issue.  R + A z at 256 x 128, p = 3: 655 us; 963 us when all
// three derivatives were traced from both sides, both viscous fluxes formed on
// every face, q_com - q subtracted at every point, a third of the face threads
// kept for walls, and 2 / h divided out by every thread.
// Element-Jacobi columns use k_ns_res after k_ns_fulltrace, which traces q and
// its whole gradient: slot = (element, column c), own state perturbed in DOF
// c by eps_c = beps (1 + |q_c|), own traces recomputed, neighbour traces
// frozen; it forms the element's four face fluxes itself and stages column c
// of shift*I - J_ee for the inversion kernel.  The unperturbed residual of the
// difference quotients comes from the same kernel (mode 0), by the same
// operations.
// In a thin wall cell the heat flux carries the rounding of D q on the total
// energy (44.6 at Mach 0.2) times (2 / h)^2, which is what limits R: the normal
// derivatives, the liftings and q_com - q keep one order of operations.
// Walls (isothermal, no slip) at the y ends: boundary state
// (rho_int, 0, 0, rho_int R T_w / (gamma - 1)), common gradient = own
// gradient + own lifting, inviscid wall flux g(q_b).  Gas constant R = 1.
#include "device.cuh"

namespace frk {
namespace {

struct NsArgs {
  const double* U;
  const double* z;
  const double* R0;
  const double* b;
  double* out;
  double* tb;          // traces [ne][4 faces][N][q 4, q_n 4]; for the blocks [ne][4][N][4 vars][q, q_x, q_y]
  double* fb;          // [ne][W, S][N][q_com 4, f_n 4], then the north wall's [nx][N][8]
  const double* hx;
  const double* hy;
  const double* sx;    // 2 / hx
  const double* sy;    // 2 / hy
  const double* eps2;
  const int* done;
  long long ne;
  int nx, ny, wall_y;
  double gam, mu, kappa, gx, t_wall;
  double shift, beps;
  Tables tab;
};

template <int P> struct NsSlots;
template <> struct NsSlots<2> { static constexpr int E = 14; };
template <> struct NsSlots<3> { static constexpr int E = 8; };
template <> struct NsSlots<4> { static constexpr int E = 5; };

template <int N>
__device__ __forceinline__ double tsum(const double* x, int stride, const double* c) {
  double s = c[0] * x[0];
#pragma unroll
  for (int k = 1; k < N; ++k) s = fma(c[k], x[k * stride], s);
  return s;
}

// viscous fluxes (f_vis, g_vis) from the state and its gradients, R = 1
__device__ __forceinline__ void visc_flux(const double q[4], const double qx[4], const double qy[4],
                                          double gam, double mu, double kappa, double fv[4],
                                          double gv[4]) {
  const double rinv = 1.0 / q[0];
  const double u = q[1] * rinv, v = q[2] * rinv, e = q[3] * rinv;
  const double ux = (qx[1] - u * qx[0]) * rinv, vx = (qx[2] - v * qx[0]) * rinv;
  const double uy = (qy[1] - u * qy[0]) * rinv, vy = (qy[2] - v * qy[0]) * rinv;
  const double Tx = (gam - 1.0) * ((qx[3] - e * qx[0]) * rinv - (u * ux + v * vx));
  const double Ty = (gam - 1.0) * ((qy[3] - e * qy[0]) * rinv - (u * uy + v * vy));
  const double div = ux + vy;
  const double txx = mu * (2.0 * ux - (2.0 / 3.0) * div);
  const double tyy = mu * (2.0 * vy - (2.0 / 3.0) * div);
  const double txy = mu * (uy + vx);
  fv[0] = 0.0; fv[1] = txx; fv[2] = txy; fv[3] = u * txx + v * txy + kappa * Tx;
  gv[0] = 0.0; gv[1] = txy; gv[2] = tyy; gv[3] = u * txy + v * tyy + kappa * Ty;
}

// Shared per-element work: state into sq, reference-space derivatives into
// dxi / deta, traces (q, q_x, q_y) of face point (face, k) into t[v][3].
template <int N>
__device__ __forceinline__ void face_trace(const double* sq, const double* dxi, const double* deta,
                                           int face, int k, double sx, double sy, const double* lm,
                                           const double* lp, double t[4][3]) {
  constexpr int NP = N * N;
  const int off = face < 2 ? N * k : k;
  const int stride = face < 2 ? 1 : N;
  const double* c = (face == 0 || face == 2) ? lm : lp;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    t[v][0] = tsum<N>(sq + v * NP + off, stride, c);
    t[v][1] = sx * tsum<N>(dxi + v * NP + off, stride, c);
    t[v][2] = sy * tsum<N>(deta + v * NP + off, stride, c);
  }
}

// traces of the unperturbed state and of its gradient, for the block columns
template <int P>
__global__ void __launch_bounds__(256) k_ns_fulltrace(const NsArgs a) {
  constexpr int N = P + 1, NP = N * N, E = NsSlots<P>::E;
  __shared__ double sq[E][4 * NP], dxi[E][4 * NP], deta[E][4 * NP];
  __shared__ double sD[N][N], slm[N], slp[N];
  if (threadIdx.x < N * N) sD[threadIdx.x / N][threadIdx.x % N] = a.tab.D[threadIdx.x / N][threadIdx.x % N];
  if (threadIdx.x < N) {
    slm[threadIdx.x] = a.tab.lm[threadIdx.x];
    slp[threadIdx.x] = a.tab.lp[threadIdx.x];
  }
  const int el = threadIdx.x / NP, t = threadIdx.x % NP;
  const long long e = (long long)blockIdx.x * E + el;
  const bool active = el < E && e < a.ne;
  if (active) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long o = e * 4 * NP + v * NP + t;
      sq[el][v * NP + t] = a.U[o];
    }
  }
  __syncthreads();
  if (active) {
    const int i = t % N, j = t / N;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      double d1 = 0.0, d2 = 0.0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        d1 = fma(sD[i][k], sq[el][v * NP + k + N * j], d1);
        d2 = fma(sD[j][k], sq[el][v * NP + i + N * k], d2);
      }
      dxi[el][v * NP + t] = d1;
      deta[el][v * NP + t] = d2;
    }
  }
  __syncthreads();
  if (!active) return;
  const int ix = (int)(e % a.nx), iy = (int)(e / a.nx);
  const double sx = a.sx[ix], sy = a.sy[iy];
  for (int fp = t; fp < 4 * N; fp += NP) {
    const int face = fp / N, k = fp % N;
    double tr[4][3];
    face_trace<N>(sq[el], dxi[el], deta[el], face, k, sx, sy, slm, slp, tr);
    double* dst = a.tb + (((e * 4 + face) * N + k) * 4) * 3;
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
      for (int c = 0; c < 3; ++c) dst[v * 3 + c] = tr[v][c];
  }
}

// (block columns) common total flux across a face from the left (-) and right (+) data;
// dir 0: x-face (normal +x), 1: y-face (normal +y); hm, hp: element sizes
// normal to the face; cbr2 = (P+1)(P+2)/2.
__device__ __forceinline__ void common_flux(const double m[4][3], const double pp[4][3], int dir,
                                            double hm, double hp, double cbr2, const NsArgs& a,
                                            double qc[4], double fn[4]) {
  double qm[4], qp[4], gxc[4], gyc[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    qm[v] = m[v][0];
    qp[v] = pp[v][0];
    qc[v] = 0.5 * (qm[v] + qp[v]);
    const double rm = (2.0 / hm) * cbr2 * (qc[v] - qm[v]);   // lifting of the (-) element
    const double rp = -(2.0 / hp) * cbr2 * (qc[v] - qp[v]);  // lifting of the (+) element
    if (dir == 0) {
      gxc[v] = 0.5 * ((m[v][1] + rm) + (pp[v][1] + rp));
      gyc[v] = 0.5 * (m[v][2] + pp[v][2]);
    } else {
      gxc[v] = 0.5 * (m[v][1] + pp[v][1]);
      gyc[v] = 0.5 * ((m[v][2] + rm) + (pp[v][2] + rp));
    }
  }
  double fi[4], fv[4], gv[4];
  rusanov(qm, qp, dir, a.gam, fi);
  visc_flux(qc, gxc, gyc, a.gam, a.mu, a.kappa, fv, gv);
#pragma unroll
  for (int v = 0; v < 4; ++v) fn[v] = fi[v] - (dir == 0 ? fv[v] : gv[v]);
}

// wall face: own data o (the element is (+) on the south wall, (-) on the north wall)
__device__ __forceinline__ void wall_flux(const double o[4][3], bool south, double h, double cbr2,
                                          const NsArgs& a, double qc[4], double fn[4]) {
  double qo[4], gxc[4], gyc[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) qo[v] = o[v][0];
  qc[0] = qo[0];
  qc[1] = 0.0;
  qc[2] = 0.0;
  qc[3] = qo[0] * a.t_wall / (a.gam - 1.0);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double r = (south ? -1.0 : 1.0) * (2.0 / h) * cbr2 * (qc[v] - qo[v]);
    gxc[v] = o[v][1];
    gyc[v] = o[v][2] + r;
  }
  double f[4], g[4], fv[4], gv[4];
  euler_fluxes(qc, a.gam, f, g);
  visc_flux(qc, gxc, gyc, a.gam, a.mu, a.kappa, fv, gv);
#pragma unroll
  for (int v = 0; v < 4; ++v) fn[v] = g[v] - gv[v];
}

template <int P, int MODE>
__global__ void __launch_bounds__(256) k_ns_res(const NsArgs a) {
  constexpr int N = P + 1, NP = N * N, E = NsSlots<P>::E, NB = 4 * NP;
  static_assert(MODE == 0 || MODE == 3, "R(U) or the block columns");
  constexpr double cbr2 = (P + 1) * (P + 2) / 2.0;
  __shared__ double sq[E][4 * NP], dxi[E][4 * NP], deta[E][4 * NP];  // dxi/deta reused for F, G
  __shared__ double tr[E][4][N][4][3];   // own face traces
  __shared__ double cq[E][4][N][4];      // common solution on the own faces
  __shared__ double fnum[E][4][N][4];    // common total normal flux on the own faces
  __shared__ double sD[N][N], sDt[N][N], slm[N], slp[N], sdgL[N], sdgR[N];
  if (a.done && *a.done) return;
  if (threadIdx.x < N * N) {
    sD[threadIdx.x / N][threadIdx.x % N] = a.tab.D[threadIdx.x / N][threadIdx.x % N];
    sDt[threadIdx.x / N][threadIdx.x % N] = a.tab.Dt[threadIdx.x / N][threadIdx.x % N];
  }
  if (threadIdx.x < N) {
    slm[threadIdx.x] = a.tab.lm[threadIdx.x];
    slp[threadIdx.x] = a.tab.lp[threadIdx.x];
    sdgL[threadIdx.x] = a.tab.dgL[threadIdx.x];
    sdgR[threadIdx.x] = a.tab.dgR[threadIdx.x];
  }
  const int el = threadIdx.x / NP, t = threadIdx.x % NP;
  const long long slot = (long long)blockIdx.x * E + el;
  const long long nslots = MODE == 3 ? a.ne * NB : a.ne;
  const bool active = el < E && slot < nslots;
  const long long e = MODE == 3 ? slot / NB : slot;
  const int col = MODE == 3 ? (int)(slot % NB) : 0;
  int ix = 0, iy = 0;
  double hx = 1.0, hy = 1.0;
  double ceps = 0.0;
  if (active) {
    ix = (int)(e % a.nx);
    iy = (int)(e / a.nx);
    hx = a.hx[ix];
    hy = a.hy[iy];
    if (MODE == 3) ceps = a.beps * (1.0 + fabs(a.U[e * NB + col]));
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long o = e * 4 * NP + v * NP + t;
      double qv = a.U[o];
      if (MODE == 3 && v * NP + t == col) qv += ceps;
      sq[el][v * NP + t] = qv;
    }
  }
  __syncthreads();
  const int i = t % N, j = t / N;
  if (active) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      double d1 = 0.0, d2 = 0.0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        d1 = fma(sD[i][k], sq[el][v * NP + k + N * j], d1);
        d2 = fma(sD[j][k], sq[el][v * NP + i + N * k], d2);
      }
      dxi[el][v * NP + t] = d1;
      deta[el][v * NP + t] = d2;
    }
  }
  __syncthreads();
  const double sx = active ? a.sx[ix] : 0.0, sy = active ? a.sy[iy] : 0.0;
  if (active) {
    for (int fp = t; fp < 4 * N; fp += NP) {
      const int face = fp / N, k = fp % N;
      double o[4][3];
      face_trace<N>(sq[el], dxi[el], deta[el], face, k, sx, sy, slm, slp, o);
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int c = 0; c < 3; ++c) tr[el][face][k][v][c] = o[v][c];
    }
  }
  __syncthreads();
  // common solution, BR2 common gradient and common total flux per own face point
  if (active) {
    for (int fp = t; fp < 4 * N; fp += NP) {
      const int face = fp / N, k = fp % N;
      double o[4][3], nb[4][3], qc[4], fn[4];
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int c = 0; c < 3; ++c) o[v][c] = tr[el][face][k][v][c];
      const bool wall = a.wall_y && ((face == 2 && iy == 0) || (face == 3 && iy == a.ny - 1));
      if (wall) {
        wall_flux(o, face == 2, hy, cbr2, a, qc, fn);
      } else {
        long long nbe;
        int nface;
        double hn;
        if (face == 0) { const int jx = (ix + a.nx - 1) % a.nx; nbe = jx + (long long)a.nx * iy; nface = 1; hn = a.hx[jx]; }
        else if (face == 1) { const int jx = (ix + 1) % a.nx; nbe = jx + (long long)a.nx * iy; nface = 0; hn = a.hx[jx]; }
        else if (face == 2) { const int jy = (iy + a.ny - 1) % a.ny; nbe = ix + (long long)a.nx * jy; nface = 3; hn = a.hy[jy]; }
        else { const int jy = (iy + 1) % a.ny; nbe = ix + (long long)a.nx * jy; nface = 2; hn = a.hy[jy]; }
        const double* src = a.tb + (((nbe * 4 + nface) * N + k) * 4) * 3;
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
          for (int c = 0; c < 3; ++c) nb[v][c] = src[v * 3 + c];
        const int dir = face < 2 ? 0 : 1;
        const double hown = dir == 0 ? hx : hy;
        if (face == 0 || face == 2) common_flux(nb, o, dir, hn, hown, cbr2, a, qc, fn);
        else common_flux(o, nb, dir, hown, hn, cbr2, a, qc, fn);
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        cq[el][face][k][v] = qc[v];
        fnum[el][face][k][v] = fn[v];
      }
    }
  }
  __syncthreads();
  // corrected gradient and total flux at the own point (overwrites dxi / deta)
  if (active) {
    double q[4], gxv[4], gyv[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      q[v] = sq[el][v * NP + t];
      double dx = dxi[el][v * NP + t];
      dx = fma(cq[el][0][j][v] - tr[el][0][j][v][0], sdgL[i], dx);
      dx = fma(cq[el][1][j][v] - tr[el][1][j][v][0], sdgR[i], dx);
      double dy = deta[el][v * NP + t];
      dy = fma(cq[el][2][i][v] - tr[el][2][i][v][0], sdgL[j], dy);
      dy = fma(cq[el][3][i][v] - tr[el][3][i][v][0], sdgR[j], dy);
      gxv[v] = sx * dx;
      gyv[v] = sy * dy;
    }
    double f[4], g[4], fv[4], gv[4];
    euler_fluxes(q, a.gam, f, g);
    visc_flux(q, gxv, gyv, a.gam, a.mu, a.kappa, fv, gv);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      dxi[el][v * NP + t] = f[v] - fv[v];
      deta[el][v * NP + t] = g[v] - gv[v];
    }
  }
  __syncthreads();
  if (!active) return;
  const long long base = e * 4 * NP + t;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    double dF = sdgL[i] * fnum[el][0][j][v];
    dF = fma(sdgR[i], fnum[el][1][j][v], dF);
#pragma unroll
    for (int k = 0; k < N; ++k) dF = fma(sDt[i][k], dxi[el][v * NP + k + N * j], dF);
    double dG = sdgL[j] * fnum[el][2][i][v];
    dG = fma(sdgR[j], fnum[el][3][i][v], dG);
#pragma unroll
    for (int k = 0; k < N; ++k) dG = fma(sDt[j][k], deta[el][v * NP + i + N * k], dG);
    double R = -fma(sx, dF, sy * dG);
    if (v == 1) R = fma(sq[el][t], a.gx, R);
    if (v == 3) R = fma(sq[el][NP + t], a.gx, R);
    const long long o = base + v * NP;
    if (MODE == 0) {
      a.out[o] = R;
    } else {
      // column col of M = shift I - J_ee, staged column-major [col][row]
      const int row = v * NP + t;
      const double m = (row == col ? a.shift : 0.0) - (R - a.R0[o]) / ceps;
      a.out[(e * NB + col) * NB + row] = m;
    }
  }
}

// q and its normal derivative at the face points; work items over the CTA's
// E elements x 4N points, so no degree leaves threads with a second round alone
template <int P, bool PERTURB>
__global__ void __launch_bounds__(256) k_ns_trace(const NsArgs a) {
  constexpr int N = P + 1, NP = N * N, E = NsSlots<P>::E;
  __shared__ double sq[E][4 * NP], dd[2][E][4 * NP];
  __shared__ double sD[N][N], sl[2][N];  // l_k(-+1)
  if (a.done && *a.done) return;
  if (threadIdx.x < N * N) sD[threadIdx.x / N][threadIdx.x % N] = a.tab.D[threadIdx.x / N][threadIdx.x % N];
  if (threadIdx.x < N) {
    sl[0][threadIdx.x] = a.tab.lm[threadIdx.x];
    sl[1][threadIdx.x] = a.tab.lp[threadIdx.x];
  }
  const long long e0 = (long long)blockIdx.x * E;
  const int ne = a.ne - e0 < E ? (int)(a.ne - e0) : E;
  const double eps = PERTURB ? a.eps2[0] : 0.0;
  for (int i = threadIdx.x; i < ne * 4 * NP; i += blockDim.x) {
    const long long o = e0 * 4 * NP + i;
    sq[0][i] = PERTURB ? fma(eps, a.z[o], a.U[o]) : a.U[o];
  }
  __syncthreads();
  {
    const int el = threadIdx.x / NP, t = threadIdx.x % NP, i = t % N, j = t / N;
    if (el < ne) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        double d1 = 0.0, d2 = 0.0;
#pragma unroll
        for (int k = 0; k < N; ++k) {
          d1 = fma(sD[i][k], sq[el][v * NP + k + N * j], d1);
          d2 = fma(sD[j][k], sq[el][v * NP + i + N * k], d2);
        }
        dd[0][el][v * NP + t] = d1;
        dd[1][el][v * NP + t] = d2;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ne * 4 * N; i += blockDim.x) {
    const int el = i / (4 * N), face = (i / N) % 4, k = i % N;
    const long long e = e0 + el;
    const double s = face < 2 ? a.sx[e % a.nx] : a.sy[e / a.nx];
    const int off = face < 2 ? N * k : k, stride = face < 2 ? 1 : N;
    double* dst = a.tb + ((e * 4 + face) * N + k) * 8;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      dst[v] = tsum<N>(sq[el] + v * NP + off, stride, sl[face & 1]);
      dst[4 + v] = s * tsum<N>(dd[face >> 1][el] + v * NP + off, stride, sl[face & 1]);
    }
  }
}

// Viscous flux along a face normal from the common state, its normal gradient
// gn and tangential gradient gt (dir 0: normal x, 1: normal y), R = 1.
__device__ __forceinline__ void visc_normal(const double q[4], const double gn[4], const double gt[4], int dir,
                                            const NsArgs& a, double fv[4]) {
  const double rinv = rcp_fast(q[0]);
  const double vn = (dir == 0 ? q[1] : q[2]) * rinv, vt = (dir == 0 ? q[2] : q[1]) * rinv, e = q[3] * rinv;
  const double n_n = fma(-vn, gn[0], dir == 0 ? gn[1] : gn[2]) * rinv;  // d v_n / d n
  const double t_n = fma(-vt, gn[0], dir == 0 ? gn[2] : gn[1]) * rinv;  // d v_t / d n
  const double n_t = fma(-vn, gt[0], dir == 0 ? gt[1] : gt[2]) * rinv;
  const double t_t = fma(-vt, gt[0], dir == 0 ? gt[2] : gt[1]) * rinv;
  const double Tn = (a.gam - 1.0) * fma(-vt, t_n, fma(-vn, n_n, fma(-e, gn[0], gn[3]) * rinv));
  const double tnn = a.mu * fma(4.0 / 3.0, n_n, (-2.0 / 3.0) * t_t);
  const double tnt = a.mu * (t_n + n_t);
  fv[0] = 0.0;
  fv[1] = dir == 0 ? tnn : tnt;
  fv[2] = dir == 0 ? tnt : tnn;
  fv[3] = fma(a.kappa, Tn, fma(vt, tnt, vn * tnn));
}

// threads of k_ns_face: whole faces of N points per CTA
template <int P> struct FaceThreads { static constexpr int value = 256 / (P + 1) * (P + 1); };

// one thread per point of the west and south faces of every element, then of
// the north wall; the N threads of a face exchange its common solution in
// shared memory for the tangential derivative
template <int P>
__global__ void __launch_bounds__(256) k_ns_face(const NsArgs a) {
  constexpr int N = P + 1;
  constexpr double cbr2 = (P + 1) * (P + 2) / 2.0;
  __shared__ double sD[N][N], sc[FaceThreads<P>::value][4];
  if (a.done && *a.done) return;
  if (threadIdx.x < N * N) sD[threadIdx.x / N][threadIdx.x % N] = a.tab.D[threadIdx.x / N][threadIdx.x % N];
  const long long tid = (long long)blockIdx.x * FaceThreads<P>::value + threadIdx.x;
  const long long inner = a.ne * 2 * N;
  const bool active = tid < inner + (a.wall_y ? (long long)a.nx * N : 0);
  const bool north = tid >= inner;
  const int k = threadIdx.x % N;
  const int slot = north ? 1 : (int)((tid / N) % 2);  // 0: west face, 1: south face (or the north wall)
  const long long e = north ? a.ne - a.nx + (tid - inner) / N : tid / (2 * N);
  const int ix = (int)(e % a.nx), iy = (int)(e / a.nx);
  const bool wall = north || (slot == 1 && a.wall_y && iy == 0);
  double m[8], o[8], qc[4], gn[4], gt[4];
  double so = 0.0, sn = 0.0, st = 0.0;
  if (active) {
    const int oface = slot == 0 ? 0 : (north ? 3 : 2);
    const double* src = a.tb + ((e * 4 + oface) * N + k) * 8;
#pragma unroll
    for (int v = 0; v < 8; ++v) o[v] = src[v];
    so = slot == 0 ? a.sx[ix] : a.sy[iy];
    st = slot == 0 ? a.sy[iy] : a.sx[ix];
    if (!wall) {
      const int jx = slot == 0 ? (ix + a.nx - 1) % a.nx : ix, jy = slot == 0 ? iy : (iy + a.ny - 1) % a.ny;
      const double* nsrc = a.tb + (((jx + (long long)a.nx * jy) * 4 + (slot == 0 ? 1 : 3)) * N + k) * 8;
#pragma unroll
      for (int v = 0; v < 8; ++v) m[v] = nsrc[v];
      sn = slot == 0 ? a.sx[jx] : a.sy[jy];
    }
    // the field whose derivative along the face is the tangential gradient: the
    // common solution, at a wall the element's own trace
#pragma unroll
    for (int v = 0; v < 4; ++v) sc[threadIdx.x][v] = qc[v] = wall ? o[v] : 0.5 * (m[v] + o[v]);
  }
  __syncthreads();
  if (!active) return;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double* x = &sc[threadIdx.x - k][v];
    double s = sD[k][0] * x[0];
#pragma unroll
    for (int l = 1; l < N; ++l) s = fma(sD[k][l], x[4 * l], s);
    gt[v] = st * s;
  }
  double fi[4], fv[4];
  if (wall) {
    double f[4];
    qc[1] = qc[2] = 0.0;
    qc[3] = qc[0] * a.t_wall / (a.gam - 1.0);
#pragma unroll
    for (int v = 0; v < 4; ++v)  // the lifting points out of the wall
      gn[v] = o[4 + v] + (north ? 1.0 : -1.0) * so * cbr2 * (qc[v] - o[v]);
    euler_fluxes(qc, a.gam, f, fi);
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const double rm = sn * cbr2 * (qc[v] - m[v]);   // lifting of the (-) element
      const double rp = -so * cbr2 * (qc[v] - o[v]);  // lifting of the (+) element
      gn[v] = 0.5 * ((m[4 + v] + rm) + (o[4 + v] + rp));
    }
    rusanov2<false>(m, o, slot, a.gam, fi);
#pragma unroll
    for (int v = 0; v < 4; ++v) fi[v] *= 0.5;
  }
  visc_normal(qc, gn, gt, slot, a, fv);
  double* dst = a.fb + (north ? inner * 8 + (tid - inner) * 8 : tid * 8);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    dst[v] = qc[v];
    dst[4 + v] = fi[v] - fv[v];
  }
}

template <int P, int MODE>
__global__ void __launch_bounds__(256) k_ns_cell(const NsArgs a) {
  constexpr int N = P + 1, NP = N * N, E = NsSlots<P>::E;
  constexpr bool PERTURB = MODE == 1 || MODE == 2;
  __shared__ double sq[E][4 * NP], dxi[E][4 * NP], deta[E][4 * NP];
  __shared__ double dq[E][4][N][4];    // q_com minus the own trace on the own faces [W,E,S,N]
  __shared__ double fnum[E][4][N][4];  // common total flux on the own faces
  __shared__ double sD[N][N], sDt[N][N], sdgL[N], sdgR[N];
  if (a.done && *a.done) return;
  if (threadIdx.x < N * N) {
    sD[threadIdx.x / N][threadIdx.x % N] = a.tab.D[threadIdx.x / N][threadIdx.x % N];
    sDt[threadIdx.x / N][threadIdx.x % N] = a.tab.Dt[threadIdx.x / N][threadIdx.x % N];
  }
  if (threadIdx.x < N) {
    sdgL[threadIdx.x] = a.tab.dgL[threadIdx.x];
    sdgR[threadIdx.x] = a.tab.dgR[threadIdx.x];
  }
  const int el = threadIdx.x / NP, t = threadIdx.x % NP;
  const long long e = (long long)blockIdx.x * E + el;
  const bool active = el < E && e < a.ne;
  double eps = 0.0, ieps = 0.0;
  if (PERTURB) {
    eps = a.eps2[0];
    ieps = a.eps2[1];
  }
  double sx = 0.0, sy = 0.0;
  if (active) {
    const int ix = (int)(e % a.nx), iy = (int)(e / a.nx);
    sx = a.sx[ix];
    sy = a.sy[iy];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const long long o = e * 4 * NP + v * NP + t;
      sq[el][v * NP + t] = PERTURB ? fma(eps, a.z[o], a.U[o]) : a.U[o];
    }
    // the common data of the four faces: W, S own; E, N the neighbours' W, S (or the wall's)
    for (int fp = t; fp < 4 * N; fp += NP) {
      const int face = fp / N, k = fp % N;
      long long fe = e * 2 + (face >> 1);
      if (face == 1) fe = ((ix + 1) % a.nx + (long long)a.nx * iy) * 2;
      else if (face == 3 && a.wall_y && iy == a.ny - 1) fe = a.ne * 2 + ix;
      else if (face == 3) fe = (ix + (long long)a.nx * ((iy + 1) % a.ny)) * 2 + 1;
      const double* fd = a.fb + (fe * N + k) * 8;
      const double* tr = a.tb + ((e * 4 + face) * N + k) * 8;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        dq[el][face][k][v] = fd[v] - tr[v];
        fnum[el][face][k][v] = fd[4 + v];
      }
    }
  }
  __syncthreads();
  const int i = t % N, j = t / N;
  // FR-corrected gradient and total flux at the own point
  if (active) {
    double q[4], gx[4], gy[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      q[v] = sq[el][v * NP + t];
      double d1 = 0.0, d2 = 0.0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        d1 = fma(sD[i][k], sq[el][v * NP + k + N * j], d1);
        d2 = fma(sD[j][k], sq[el][v * NP + i + N * k], d2);
      }
      d1 = fma(dq[el][0][j][v], sdgL[i], d1);
      d1 = fma(dq[el][1][j][v], sdgR[i], d1);
      d2 = fma(dq[el][2][i][v], sdgL[j], d2);
      d2 = fma(dq[el][3][i][v], sdgR[j], d2);
      gx[v] = sx * d1;
      gy[v] = sy * d2;
    }
    double f[4], g[4];
    euler_fluxes(q, a.gam, f, g);
    const double rinv = 1.0 / q[0];  // the one of euler_fluxes
    const double u = q[1] * rinv, w = q[2] * rinv, en = q[3] * rinv;
    const double ux = fma(-u, gx[0], gx[1]) * rinv, wx = fma(-w, gx[0], gx[2]) * rinv;
    const double uy = fma(-u, gy[0], gy[1]) * rinv, wy = fma(-w, gy[0], gy[2]) * rinv;
    const double Tx = (a.gam - 1.0) * fma(-w, wx, fma(-u, ux, fma(-en, gx[0], gx[3]) * rinv));
    const double Ty = (a.gam - 1.0) * fma(-w, wy, fma(-u, uy, fma(-en, gy[0], gy[3]) * rinv));
    const double txx = a.mu * fma(4.0 / 3.0, ux, (-2.0 / 3.0) * wy);
    const double tyy = a.mu * fma(4.0 / 3.0, wy, (-2.0 / 3.0) * ux);
    const double txy = a.mu * (uy + wx);
    double* F = dxi[el] + t;
    double* G = deta[el] + t;
    F[0] = f[0];
    F[NP] = f[1] - txx;
    F[2 * NP] = f[2] - txy;
    F[3 * NP] = f[3] - fma(a.kappa, Tx, fma(w, txy, u * txx));
    G[0] = g[0];
    G[NP] = g[1] - txy;
    G[2 * NP] = g[2] - tyy;
    G[3 * NP] = g[3] - fma(a.kappa, Ty, fma(w, tyy, u * txy));
  }
  __syncthreads();
  if (!active) return;
  const long long base = e * 4 * NP + t;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    double dF = sdgL[i] * fnum[el][0][j][v];
    dF = fma(sdgR[i], fnum[el][1][j][v], dF);
#pragma unroll
    for (int k = 0; k < N; ++k) dF = fma(sDt[i][k], dxi[el][v * NP + k + N * j], dF);
    double dG = sdgL[j] * fnum[el][2][i][v];
    dG = fma(sdgR[j], fnum[el][3][i][v], dG);
#pragma unroll
    for (int k = 0; k < N; ++k) dG = fma(sDt[j][k], deta[el][v * NP + i + N * k], dG);
    double R = -fma(sx, dF, sy * dG);
    if (v == 1) R = fma(sq[el][t], a.gx, R);
    if (v == 3) R = fma(sq[el][NP + t], a.gx, R);
    const long long o = base + v * NP;
    if (MODE == 0) {
      a.out[o] = R;
    } else {
      const double zo = a.z[o];
      const double Az = eps > 0.0 ? fma(-(R - a.R0[o]), ieps, a.shift * zo) : a.shift * zo;
      a.out[o] = MODE == 2 ? a.b[o] - Az : Az;
    }
  }
}

NsArgs make_args(fr_ctx* ctx) {
  NsArgs a{};
  a.tb = ctx->tb;
  a.fb = ctx->fb;
  a.hx = ctx->hx;
  a.hy = ctx->hy;
  a.sx = ctx->sx;
  a.sy = ctx->sy;
  a.ne = ctx->ne;
  a.nx = ctx->nx;
  a.ny = ctx->ny;
  a.wall_y = ctx->wall_y;
  a.gam = ctx->opts.gamma;
  a.mu = ctx->opts.mu;
  const double cp = ctx->opts.gamma / (ctx->opts.gamma - 1.0);  // R = 1
  a.kappa = ctx->opts.mu * cp / ctx->opts.prandtl;
  a.gx = ctx->opts.body_force_x;
  a.t_wall = ctx->opts.wall_temperature;
  a.beps = ctx->opts.block_eps_rel;
  a.tab = ctx->tab;
  return a;
}

template <int P>
int ns_launch(fr_ctx* ctx, int mode, const NsArgs& a, cudaStream_t s, double wb, double wf) {
  constexpr int NP = (P + 1) * (P + 1), E = NsSlots<P>::E;
  const unsigned gt = (unsigned)((ctx->ne + E - 1) / E);
  ProfScope ps_(ctx, mode == 0 ? FR_KF_RESIDUAL : FR_KF_JV, s, wb, wf);  // one timed record for the three kernels
  if (mode == 0) k_ns_trace<P, false><<<gt, E * NP, 0, s>>>(a);
  else k_ns_trace<P, true><<<gt, E * NP, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  count_launch();  // the scope counted the trace kernel
  const long long nf = (ctx->ne * 2 + (a.wall_y ? ctx->nx : 0)) * (P + 1);
  k_ns_face<P><<<(unsigned)((nf + FaceThreads<P>::value - 1) / FaceThreads<P>::value), FaceThreads<P>::value, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  count_launch();
  if (mode == 0) k_ns_cell<P, 0><<<gt, E * NP, 0, s>>>(a);
  else if (mode == 1) k_ns_cell<P, 1><<<gt, E * NP, 0, s>>>(a);
  else k_ns_cell<P, 2><<<gt, E * NP, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int dispatch(fr_ctx* ctx, int mode, const NsArgs& a, cudaStream_t s, double wb, double wf) {
  switch (ctx->p) {
    case 2: return ns_launch<2>(ctx, mode, a, s, wb, wf);
    case 3: return ns_launch<3>(ctx, mode, a, s, wb, wf);
    case 4: return ns_launch<4>(ctx, mode, a, s, wb, wf);
    default: return set_error(ctx, FR_ERR_UNSUPPORTED, "degree %d not compiled", ctx->p);
  }
}

// traces of U and its gradient, R(U) into ctx->rloc and the block columns into
// ctx->mst, all by the operations of k_ns_res
template <int P>
int ns_columns(fr_ctx* ctx, NsArgs a, double shift, cudaStream_t s) {
  constexpr int NP = (P + 1) * (P + 1), E = NsSlots<P>::E, NB = 4 * NP;
  const unsigned gt = (unsigned)((ctx->ne + E - 1) / E);
  ProfScope ps_(ctx, FR_KF_FACTOR, s);  // one timed record for the three kernels
  k_ns_fulltrace<P><<<gt, E * NP, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  count_launch();
  a.out = ctx->rloc;
  k_ns_res<P, 0><<<gt, E * NP, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  count_launch();
  a.R0 = ctx->rloc;
  a.out = ctx->mst;
  a.shift = shift;
  k_ns_res<P, 3><<<(unsigned)((ctx->ne * NB + E - 1) / E), E * NP, 0, s>>>(a);
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

}  // namespace

int launch_ns_residual(fr_ctx* ctx, int mode, const double* U, const double* z, const double* R0,
                       const double* b, double* out, double shift, const double* eps2,
                       const int* done, cudaStream_t s) {
  NsArgs a = make_args(ctx);
  a.U = U;
  a.z = z;
  a.R0 = R0;
  a.b = b;
  a.out = out;
  a.eps2 = eps2;
  a.done = done;
  a.shift = shift;
  // inside a GMRES cycle both kernels return at once once the cycle is done
  const double nd = (double)ctx->ndof;
  const bool in_cycle = done != nullptr;
  const double wb = in_cycle ? 0.0 : (mode == 0 ? 16.0 : (mode == 1 ? 32.0 : 40.0)) * nd;
  const double wf = in_cycle ? 0.0 : ns_residual_flops_per_element(ctx->p) * (double)ctx->ne + (mode == 0 ? 0.0 : 6.0 * nd);
  return dispatch(ctx, mode, a, s, wb, wf);
}

int launch_ns_factor(fr_ctx* ctx, const double* U, double shift, cudaStream_t s) {
  NsArgs a = make_args(ctx);
  a.U = U;
  switch (ctx->p) {
    case 2: FRK_TRY(ns_columns<2>(ctx, a, shift, s)); break;
    case 3: FRK_TRY(ns_columns<3>(ctx, a, shift, s)); break;
    case 4: FRK_TRY(ns_columns<4>(ctx, a, shift, s)); break;
    default: return set_error(ctx, FR_ERR_UNSUPPORTED, "degree %d not compiled", ctx->p);
  }
  return launch_block_invert(ctx, ctx->mst, 0.0, s);
}

}  // namespace frk
