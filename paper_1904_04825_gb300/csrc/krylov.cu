// Restarted GMRES(m) of Sec. 4.5 on the device.
//
// Arnoldi uses classical Gram-Schmidt with one re-orthogonalisation pass
// (CGS2): every pass is one multi-dot kernel and one multi-AXPY kernel over
// the whole basis slice, with deterministic two-stage reductions.  The
// Hessenberg column, the Givens rotation and the convergence test run in a
// one-warp kernel, so a cycle of m iterations is launched without any host
// round trip: once the device sets `done`, the remaining kernels of the
// cycle return at once.  The host reads the cycle status once per restart.
#include <cmath>

#include "cycle.h"
#include "krylov_body.cuh"

namespace frk {
namespace {

unsigned vgrid(const fr_ctx* ctx, long long n) {
  long long g = (n + kThreads - 1) / kThreads;
  if (g > ctx->vec_blocks) g = ctx->vec_blocks;
  return (unsigned)(g < 1 ? 1 : g);
}

__global__ void k_sumsq(const double* __restrict__ x, long long n, double* out, Reduce red,
                        EpsArgs ea) {
  __shared__ double sh[32];
  const double bs = block_sum(sumsq_rows(x, n, blockIdx.x, gridDim.x), sh);
  if (threadIdx.x == 0) red.value(0)[blockIdx.x] = bs;
  if (last_block(red.counter)) {
    finish_sums(red, 1, out);
    if (threadIdx.x == 0) write_eps(ea, *out);
  }
}

// out[0] = ||x||^2 (the FD step's ||U||^2), out[1] = ||y||^2 and the FD step from
// both: one launch for the two norms of a product, each summed as k_sumsq sums it
__global__ void k_sumsq2(const double* __restrict__ x, const double* __restrict__ y, long long n, double* out,
                         Reduce red, EpsArgs ea) {
  __shared__ double sh[32];
  const double bx = block_sum(sumsq_rows(x, n, blockIdx.x, gridDim.x), sh);
  const double by = block_sum(sumsq_rows(y, n, blockIdx.x, gridDim.x), sh);
  if (threadIdx.x == 0) {
    red.value(0)[blockIdx.x] = bx;
    red.value(1)[blockIdx.x] = by;
  }
  if (last_block(red.counter)) {
    static_assert(kNormValues == 2, "the scratch of fr_jv_noalloc holds the columns written here");
    finish_sums(red, kNormValues, out);
    __syncthreads();
    if (threadIdx.x == 0) write_eps(ea, out[1]);
  }
}

struct Lincomb {
  const double* x[8];
  double c[8];
  int n;
};

// out = sum_t c_t x_t (out may alias any x_t), optional sum of squares of out
__global__ void k_lincomb(double* out, long long len, const Lincomb lc, double* sumsq, Reduce red) {
  __shared__ double sh[32];
  double ss = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < len;
       i += (long long)gridDim.x * blockDim.x) {
    double v = lc.c[0] * lc.x[0][i];
    for (int t = 1; t < lc.n; ++t) v = fma(lc.c[t], lc.x[t][i], v);
    out[i] = v;
    ss = fma(v, v, ss);
  }
  if (sumsq) {
    const double bs = block_sum(ss, sh);
    if (threadIdx.x == 0) red.value(0)[blockIdx.x] = bs;
    if (last_block(red.counter)) finish_sums(red, 1, sumsq);
  }
}

__global__ void __launch_bounds__(256) k_dots(const double* __restrict__ V, long long ldv, int nvec,
                                              const double* __restrict__ w, long long n, double* out,
                                              int with_self, Reduce red, const int* done,
                                              const int* gate) {
  dots_body(V, ldv, nvec, w, n, out, with_self, red, done, gate, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256) k_update(double* __restrict__ w, const double* __restrict__ V,
                                                long long ldv, int nvec, const double* h,
                                                long long n, double* sumsq, Reduce red,
                                                const int* done, const int* gate, Reorth ro) {
  update_body(w, V, ldv, nvec, h, n, sumsq, red, done, gate, ro, blockIdx.x, gridDim.x);
}

// start of a cycle: beta = ||r||, g = beta e_1, done if beta <= rtol ||b||
__global__ void k_cycle_init(GmresDev gd, const double* nr2, const double* nb2, double rtol, int m,
                             const int* fin) {
  if (threadIdx.x != 0) return;
  if (fin && *fin) {  // solve already finished: the whole cycle is skipped
    *gd.k = 0;
    *gd.done = 1;
    return;
  }
  const double beta = sqrt(*nr2);
  const double target = rtol * sqrt(*nb2);
  for (int i = 0; i <= m; ++i) gd.g[i] = 0.0;
  gd.g[0] = beta;
  *gd.target = target;
  *gd.res = beta;
  *gd.k = 0;
  *gd.done = (beta <= target) ? 1 : 0;
  for (int i = 0; i < m; ++i) gd.rflag[i] = 0;
  gd.invh[0] = beta > 0.0 ? 1.0 / beta : 0.0;
}

__global__ void k_givens(GmresDev gd, int j, const double* nw2) {
  givens_body(gd, j, nw2);
}

__global__ void k_backsub(GmresDev gd) {
  __shared__ double Hs[kTriangle], ys[kMaxVec];
  const int k = *gd.k;
  backsub(gd, k, Hs, ys);
  for (int i = threadIdx.x; i < k; i += blockDim.x) gd.y[i] = ys[i];
}

// cycle status for the host: [k, |g_k|, rtol ||b||, ||b||]; marks the
// solve finished once the residual met the target
__global__ void k_status(GmresDev gd, const double* nb2, double* out, int* fin, const int* kerr) {
  if (threadIdx.x != 0) return;
  if (*kerr) {  // a bounded wait gave up in this cycle
    out[0] = -1.0;
    return;
  }
  if (fin) {
    if (*fin) {
      out[0] = 0.0;
      return;
    }
    if (*gd.res <= *gd.target) *fin = 1;
  }
  out[0] = (double)*gd.k;
  out[1] = *gd.res;
  out[2] = *gd.target;
  out[3] = sqrt(*nb2);
}

__global__ void k_copy(double* dst, const double* src, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

__global__ void k_fill(double* dst, double v, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = v;
}

// ---- batched Arnoldi-step kernels: the CTAs of every instance in one grid,
// instance k owning blocks [start[k], start[k+1]) (the same partition as its
// single-instance launch, so every reduction sums in the same order) ----
__global__ void __launch_bounds__(256) kb_dots(const BatchKrylov* __restrict__ tab, const int* __restrict__ start,
                                               int ninst, int j, int second) {
  const int k = batch_instance(start, ninst, blockIdx.x);
  const BatchKrylov& t = tab[k];
  const int bid = blockIdx.x - start[k], nblk = start[k + 1] - start[k];
  const long long n = t.n;
  dots_body(t.V, n, j + 1, t.V + (size_t)(j + 1) * n, n, second ? t.gd.h2 : t.gd.h1, second ? 0 : 1, t.red,
            t.gd.done, second ? t.gd.rflag + j : nullptr, bid, nblk);
}

__global__ void __launch_bounds__(256) kb_update(const BatchKrylov* __restrict__ tab, const int* __restrict__ start,
                                                 int ninst, int j, int second) {
  const int k = batch_instance(start, ninst, blockIdx.x);
  const BatchKrylov& t = tab[k];
  const int bid = blockIdx.x - start[k], nblk = start[k + 1] - start[k];
  const long long n = t.n;
  const Reorth none{nullptr, 0.0, nullptr, nullptr};
  const Reorth first{t.gd.h1 + (j + 1), t.eta2, t.gd.rflag + j, t.gd.h2};
  update_body(t.V + (size_t)(j + 1) * n, t.V, n, j + 1, second ? t.gd.h2 : t.gd.h1, n, t.nw2, t.red, t.gd.done,
              second ? t.gd.rflag + j : nullptr, second ? none : first, bid, nblk);
}

__global__ void kb_givens(const BatchKrylov* __restrict__ tab, int j) {
  const BatchKrylov& t = tab[blockIdx.x];
  givens_body(t.gd, j, t.nw2);
}

}  // namespace

BatchKrylov batch_krylov_args(fr_ctx* ctx) {
  BatchKrylov t;
  t.V = ctx->V;
  t.n = ctx->ndof;
  t.gd = ctx->gd;
  t.red = ctx->red;
  t.nw2 = ctx->scal + S_NW2;
  t.eta2 = ctx->opts.reorth_eta * ctx->opts.reorth_eta;
  return t;
}

unsigned vec_grid_of(const fr_ctx* ctx) { return vgrid(ctx, ctx->ndof); }

// The Gram-Schmidt passes and the Givens step of Arnoldi iteration j of every
// instance of a batch: tab / start describe the instances (device arrays),
// nblocks = start[ninst].
int launch_batch_gs_givens(const BatchKrylov* tab, const int* start, int ninst, int nblocks, int j, cudaStream_t s) {
  count_launches(5);
  kb_dots<<<nblocks, kThreads, 0, s>>>(tab, start, ninst, j, 0);
  kb_update<<<nblocks, kThreads, 0, s>>>(tab, start, ninst, j, 0);
  kb_dots<<<nblocks, kThreads, 0, s>>>(tab, start, ninst, j, 1);
  kb_update<<<nblocks, kThreads, 0, s>>>(tab, start, ninst, j, 1);
  kb_givens<<<ninst, 32, 0, s>>>(tab, j);
  return cudaGetLastError() == cudaSuccess ? FR_OK : FR_ERR_CUDA;
}

EpsArgs eps_args(fr_ctx* ctx, bool on) {
  EpsArgs ea{ctx->scal + S_NU2, ctx->opts.eps_rel, ctx->opts.eps_fixed, on ? ctx->scal + S_EPS : nullptr};
  return ea;
}

int launch_sumsq(fr_ctx* ctx, const double* x, double* out, cudaStream_t s, bool with_eps) {
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_sumsq<<<vgrid(ctx, ctx->ndof), kThreads, 0, s>>>(x, ctx->ndof, out, ctx->red, eps_args(ctx, with_eps)); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int launch_norms_eps(fr_ctx* ctx, const double* U, const double* z, cudaStream_t s) {
  static_assert(S_NZ2 == S_NU2 + 1, "k_sumsq2 writes the two norms side by side");
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_sumsq2<<<vgrid(ctx, ctx->ndof), kThreads, 0, s>>>(U, z, ctx->ndof, ctx->scal + S_NU2, ctx->red, eps_args(ctx, true)); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int launch_lincomb(fr_ctx* ctx, double* out, int nterms, const double* const* xs,
                   const double* coefs, double* sumsq, cudaStream_t s) {
  if (nterms < 1 || nterms > 8) return set_error(ctx, FR_ERR_INVALID_ARG, "lincomb of %d terms", nterms);
  Lincomb lc{};
  lc.n = nterms;
  for (int t = 0; t < nterms; ++t) {
    lc.x[t] = xs[t];
    lc.c[t] = coefs[t];
  }
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_lincomb<<<vgrid(ctx, ctx->ndof), kThreads, 0, s>>>(out, ctx->ndof, lc, sumsq, ctx->red); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int launch_copy(fr_ctx* ctx, double* dst, const double* src, cudaStream_t s) {
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_copy<<<vgrid(ctx, ctx->ndof), kThreads, 0, s>>>(dst, src, ctx->ndof); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int launch_fill(fr_ctx* ctx, double* dst, double v, cudaStream_t s) {
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_fill<<<vgrid(ctx, ctx->ndof), kThreads, 0, s>>>(dst, v, ctx->ndof); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

// One whole GMRES cycle enqueued without any host synchronisation (for CUDA
// graph capture): r = b - A x (exactly b for x = 0), m Arnoldi iterations
// that stop on the device, the solution update, and the status
// [k, |g_k|, target, ||b||] written to status (device, 4 doubles).  The three
// parts are also enqueued separately by batches, whose Arnoldi iterations
// run as batched launches over all instances.
int gmres_cycle_prologue(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b,
                         double* x, int m, double rtol, int* fin, cudaStream_t s) {
  double* sc = ctx->scal;
  FRK_TRY(launch_linearize(ctx, U, s));
  FRK_TRY(launch_sumsq(ctx, U, sc + S_NU2, s));
  FRK_TRY(launch_sumsq(ctx, b, sc + S_NB2, s));
  FRK_TRY(launch_sumsq(ctx, x, sc + S_NZ2, s, true));
  FRK_TRY(launch_residual(ctx, 2, U, x, R0, b, ctx->V, shift, sc + S_EPS, fin, s));
  FRK_TRY(launch_sumsq(ctx, ctx->V, sc + S_NR2, s));
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_cycle_init<<<1, 32, 0, s>>>(ctx->gd, sc + S_NR2, sc + S_NB2, rtol, m, fin); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int gmres_cycle_epilogue(fr_ctx* ctx, double* x, double* status, int* fin, cudaStream_t s) {
  GmresDev& gd = ctx->gd;
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_backsub<<<1, 256, 0, s>>>(gd); }
  FRK_LAUNCHED(ctx);
  FRK_TRY(launch_solution_update(ctx, x, s));
  { ProfScope ps_(ctx, FR_KF_OTHER, s); k_status<<<1, 32, 0, s>>>(gd, ctx->scal + S_NB2, status, fin, ctx->kerr); }
  FRK_LAUNCHED(ctx);
  return FR_OK;
}

int gmres_cycle_enqueue(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b,
                        double* x, int m, double rtol, double* status, int* fin, cudaStream_t s) {
  const long long n = ctx->ndof;
  double* sc = ctx->scal;
  GmresDev& gd = ctx->gd;
  double* V = ctx->V;
  FRK_TRY(gmres_cycle_prologue(ctx, U, R0, shift, b, x, m, rtol, fin, s));
  for (int j = 0; j < m; ++j) {
    double* vj = V + (size_t)j * n;
    double* w = V + (size_t)(j + 1) * n;
    FRK_TRY(launch_block_apply(ctx, vj, gd.invh + j, ctx->z, sc + S_NZ2, gd.done, s, true));
    FRK_TRY(launch_residual(ctx, 1, U, ctx->z, R0, nullptr, w, shift, sc + S_EPS, gd.done, s));
    const Reorth none{nullptr, 0.0, nullptr, nullptr};
    const Reorth first{gd.h1 + (j + 1), ctx->opts.reorth_eta * ctx->opts.reorth_eta, gd.rflag + j, gd.h2};
    { ProfScope ps_(ctx, FR_KF_DOTS, s); k_dots<<<vgrid(ctx, n), kThreads, 0, s>>>(V, n, j + 1, w, n, gd.h1, 1, ctx->red, gd.done, nullptr); }
    { ProfScope ps_(ctx, FR_KF_UPDATE, s); k_update<<<vgrid(ctx, n), kThreads, 0, s>>>(w, V, n, j + 1, gd.h1, n, sc + S_NW2, ctx->red, gd.done, nullptr, first); }
    { ProfScope ps_(ctx, FR_KF_DOTS, s); k_dots<<<vgrid(ctx, n), kThreads, 0, s>>>(V, n, j + 1, w, n, gd.h2, 0, ctx->red, gd.done, gd.rflag + j); }
    { ProfScope ps_(ctx, FR_KF_UPDATE, s); k_update<<<vgrid(ctx, n), kThreads, 0, s>>>(w, V, n, j + 1, gd.h2, n, sc + S_NW2, ctx->red, gd.done, gd.rflag + j, none); }
    { ProfScope ps_(ctx, FR_KF_OTHER, s); k_givens<<<1, 32, 0, s>>>(gd, j, sc + S_NW2); }
    FRK_LAUNCHED(ctx);
  }
  return gmres_cycle_epilogue(ctx, x, status, fin, s);
}

// Solves of 2D Euler contexts with element blocks and up to kCycleMaxDof unknowns
// run as one launch; per-family timing and the apply's wait test need the
// separate launches.  The line lies where the launches stop costing more than the
// barriers: a ROW3 step at p = 3 takes 10.7 ms against 11.9 ms by launches at
// 102,400 unknowns, 29.8 against 29.5 ms (BF16) and 38.8 against 38.3 ms (FP64
// blocks) at 262,144, and 170 against 131 ms at 1,638,400, where the staged apply
// and four CTAs per SM win; the 14,400-unknown ROW2 step takes 2.9 against 5.2 ms.
constexpr long long kCycleMaxDof = 200000;

bool solves_in_one_launch(const fr_ctx* ctx, int m) {
  return m + 1 <= kCycleDots &&  // <V_i, w> of up to m vectors and <w, w>
         !ctx->dim3 && !ctx->viscous && ctx->opts.jv_precision == 0 && ctx->opts.precond && ctx->p >= 2 && ctx->p <= 4 &&
         ctx->ndof <= kCycleMaxDof && ctx->prof.mask == 0 && !ctx->test_skip_copy && cycle_grid(ctx) > 0;
}

// one CTA per SM while a barrier costs more than the phases between, two above
// (14,400 unknowns: 2.9 against 3.5 ms; 102,400: 11.0 against 10.7 ms)
int cycle_grid(const fr_ctx* ctx) {
  int occ = 0;
  switch (ctx->opts.block_precision) {
    case 1: occ = resident_cycle_f32(ctx->opts.riemann, ctx->device); break;
    case 2: occ = resident_cycle_bf16(ctx->opts.riemann, ctx->device); break;
    default: occ = resident_cycle_f64(ctx->opts.riemann, ctx->device); break;
  }
  const int want = ctx->ndof <= 60000 ? 1 : 2;
  return (occ < want ? occ : want) * ctx->num_sms;
}

int launch_cycle(int prec, const CycleArgs& a, int nblocks, int riemann, cudaStream_t s) {
  switch (prec) {
    case 1: return launch_cycle_f32(a, nblocks, riemann, s);
    case 2: return launch_cycle_bf16(a, nblocks, riemann, s);
    default: return launch_cycle_f64(a, nblocks, riemann, s);
  }
}

int fill_cycle_args(fr_ctx* ctx, const double* U, const double* R0, double shift, double rtol, int m, int max_restarts,
                    CycleArgs* a) {
  *a = CycleArgs{};
  a->res = residual_args(ctx, U, R0, shift);
  a->p = ctx->p;
  a->small_tile = residual_small_tile(ctx);
  a->Minv = ctx->blocks;
  a->V = ctx->V;
  a->z = ctx->z;
  a->n = ctx->ndof;
  a->ne = ctx->ne;
  a->red = ctx->red;
  a->gd = ctx->gd;
  a->eta2 = ctx->opts.reorth_eta * ctx->opts.reorth_eta;
  a->rtol = rtol;
  a->m = m;
  a->max_restarts = max_restarts;
  a->vgrid = (int)vgrid(ctx, ctx->ndof);
  a->agrid = (int)apply_grid_of(ctx);
  a->bar = ctx->cyc_bar;
  a->polls = ctx->wait_polls < 1u << 30 ? 4 * ctx->wait_polls : ~0u;  // phases are longer than copies
  a->err = ctx->kerr;
  a->status = ctx->h_cyc;
  return a->agrid > 0 ? FR_OK : FR_ERR_UNSUPPORTED;
}

int launch_solve(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b, double* x, int m,
                 double rtol, int max_restarts, bool x_is_zero, cudaStream_t s) {
  CycleArgs a;
  FRK_TRY(fill_cycle_args(ctx, U, R0, shift, rtol, m, max_restarts, &a));
  a.b = b;
  a.x = x;
  a.x_zero = x_is_zero;
  if (launch_cycle(ctx->opts.block_precision, a, cycle_grid(ctx), ctx->opts.riemann, s) !=
      FR_OK)
    return set_error(ctx, FR_ERR_CUDA, "launch of the solve failed: %s", cudaGetErrorString(cudaGetLastError()));
  return FR_OK;
}

namespace {
int gmres_one_launch(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b, double* x, int m,
                     double rtol, int max_restarts, bool x_is_zero, fr_gmres_info* info, cudaStream_t s) {
  ctx->h_cyc->err = 1;
  FRK_TRY(launch_solve(ctx, U, R0, shift, b, x, m, rtol, max_restarts, x_is_zero, s));
  FRK_CUDA(ctx, cudaStreamSynchronize(s));
  const CycleStatus& st = *ctx->h_cyc;
  if (st.err) {  // a wait of this launch, or of an inversion or apply before it
    // CTAs that left a barrier early leave its counter anywhere
    FRK_CUDA(ctx, cudaMemsetAsync(ctx->cyc_bar, 0, sizeof(unsigned), s));
    FRK_CUDA(ctx, cudaStreamSynchronize(s));
    return set_error(ctx, FR_ERR_TIMEOUT, "a kernel's bounded wait gave up");
  }
  fr_gmres_info loc{};
  loc.iters = st.iters;
  loc.relres = st.relres;
  if (st.state == kCycleNonFinite) {
    if (info) *info = loc;
    return set_error(ctx, FR_ERR_NONFINITE, "GMRES residual is not finite");
  }
  loc.restarts = st.restarts;
  loc.converged = st.state == kCycleConverged;
  if (info) *info = loc;
  if (!loc.converged)
    return set_error(ctx, FR_ERR_NOT_CONVERGED, "GMRES stopped after %d iterations at relres %.3e", loc.iters, loc.relres);
  return FR_OK;
}
}  // namespace

int gmres_impl(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b,
               double* x, int m, double rtol, int max_restarts, bool x_is_zero,
               fr_gmres_info* info, cudaStream_t s) {
  if (solves_in_one_launch(ctx, m))
    return gmres_one_launch(ctx, U, R0, shift, b, x, m, rtol, max_restarts, x_is_zero, info, s);
  const long long n = ctx->ndof;
  double* sc = ctx->scal;
  GmresDev& gd = ctx->gd;
  double* V = ctx->V;
  fr_gmres_info loc{};
  FRK_TRY(launch_linearize(ctx, U, s));
  // ||U|| for the FD step, ||b|| for the stopping test
  FRK_TRY(launch_sumsq(ctx, U, sc + S_NU2, s));
  FRK_TRY(launch_sumsq(ctx, b, sc + S_NB2, s));
  if (!x_is_zero) {
    FRK_TRY(launch_sumsq(ctx, x, sc + S_NX2, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_scal, sc + S_NB2, sizeof(double), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_scal + 1, sc + S_NX2, sizeof(double),
                                  cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaStreamSynchronize(s));
    if (ctx->h_scal[0] == 0.0) {  // b = 0: the solution is x = 0
      FRK_TRY(launch_fill(ctx, x, 0.0, s));
      loc.converged = 1;
      if (info) *info = loc;
      return FR_OK;
    }
    x_is_zero = ctx->h_scal[1] == 0.0;
  }
  int cycles_iterated = 0;
  int status = FR_ERR_NOT_CONVERGED;
  for (int cycle = 0; cycle <= max_restarts; ++cycle) {
    // r = b - A x into V[0]
    if (cycle == 0 && x_is_zero) {
      FRK_TRY(launch_copy(ctx, V, b, s));
    } else {
      FRK_TRY(launch_sumsq(ctx, x, sc + S_NZ2, s, true));
      FRK_TRY(launch_residual(ctx, 2, U, x, R0, b, V, shift, sc + S_EPS, nullptr, s));
    }
    FRK_TRY(launch_sumsq(ctx, V, sc + S_NR2, s));
    { ProfScope ps_(ctx, FR_KF_OTHER, s); k_cycle_init<<<1, 32, 0, s>>>(gd, sc + S_NR2, sc + S_NB2, rtol, m, nullptr); }
    FRK_LAUNCHED(ctx);
    // Launch the cycle in chunks of kChunk iterations; after launching chunk
    // c, wait for the finished-flag copied after chunk c-1, so the device
    // always has queued work and at most one chunk runs past convergence.
    constexpr int kChunk = 4;
    int launched = 0, chunk = 0;
    while (launched < m) {
      const int jend = launched + kChunk < m ? launched + kChunk : m;
      for (int j = launched; j < jend; ++j) {
        double* vj = V + (size_t)j * n;
        double* w = V + (size_t)(j + 1) * n;
        // v_j = r_j / ||r_j|| (written back), z = M^{-1} v_j, ||z||^2
        FRK_TRY(launch_block_apply(ctx, vj, gd.invh + j, ctx->z, sc + S_NZ2, gd.done, s, true));
        // w = A z
        FRK_TRY(launch_residual(ctx, 1, U, ctx->z, R0, nullptr, w, shift, sc + S_EPS, gd.done, s));
        // Gram-Schmidt: one classical pass, a second one only when the
        // first shrank ||w|| below reorth_eta ||w|| (decided on the device)
        const Reorth none{nullptr, 0.0, nullptr, nullptr};
        const Reorth first{gd.h1 + (j + 1), ctx->opts.reorth_eta * ctx->opts.reorth_eta, gd.rflag + j, gd.h2};
        { ProfScope ps_(ctx, FR_KF_DOTS, s); k_dots<<<vgrid(ctx, n), kThreads, 0, s>>>(V, n, j + 1, w, n, gd.h1, 1, ctx->red, gd.done, nullptr); }
        { ProfScope ps_(ctx, FR_KF_UPDATE, s); k_update<<<vgrid(ctx, n), kThreads, 0, s>>>(w, V, n, j + 1, gd.h1, n, sc + S_NW2, ctx->red, gd.done, nullptr, first); }
        { ProfScope ps_(ctx, FR_KF_DOTS, s); k_dots<<<vgrid(ctx, n), kThreads, 0, s>>>(V, n, j + 1, w, n, gd.h2, 0, ctx->red, gd.done, gd.rflag + j); }
        { ProfScope ps_(ctx, FR_KF_UPDATE, s); k_update<<<vgrid(ctx, n), kThreads, 0, s>>>(w, V, n, j + 1, gd.h2, n, sc + S_NW2, ctx->red, gd.done, gd.rflag + j, none); }
        { ProfScope ps_(ctx, FR_KF_OTHER, s); k_givens<<<1, 32, 0, s>>>(gd, j, sc + S_NW2); }
        FRK_LAUNCHED(ctx);
      }
      launched = jend;
      const int slot = chunk & 1;
      FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_stat + 2 + slot, gd.done, sizeof(int), cudaMemcpyDeviceToHost, s));
      FRK_CUDA(ctx, cudaEventRecord(ctx->chunk_ev[slot], s));
      ++chunk;
      if (chunk >= 2) {
        const int prev = (chunk - 2) & 1;
        FRK_CUDA(ctx, cudaEventSynchronize(ctx->chunk_ev[prev]));
        if (ctx->h_stat[2 + prev]) break;
      }
    }
    { ProfScope ps_(ctx, FR_KF_OTHER, s); k_backsub<<<1, 256, 0, s>>>(gd); }
    FRK_LAUNCHED(ctx);
    FRK_TRY(launch_solution_update(ctx, x, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_stat, gd.k, sizeof(int), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_stat + 4, gd.rflag, m * sizeof(int), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_scal, gd.res, sizeof(double), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_scal + 1, gd.target, sizeof(double), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_scal + 2, sc + S_NB2, sizeof(double), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaMemcpyAsync(ctx->h_stat + 1, ctx->kerr, sizeof(int), cudaMemcpyDeviceToHost, s));
    FRK_CUDA(ctx, cudaStreamSynchronize(s));
    if (ctx->h_stat[1]) return set_error(ctx, FR_ERR_TIMEOUT, "a kernel's bounded wait for its copies gave up");
    const int k = ctx->h_stat[0];
    const double res = ctx->h_scal[0], target = ctx->h_scal[1], bn = std::sqrt(ctx->h_scal[2]);
    {  // launches of this cycle that found it finished (for per-launch timing),
       // and the algorithmic work of the k iterations that ran: apply (blocks +
       // r in, r and z out), A z (U, z, R0 in, w out), CGS2 (two multi-dots
       // reading j+1 basis vectors and w, two updates reading them and
       // reading/writing w)
      const long long sk = launched - k;
      const double nd = (double)n;
      long long second = 0;
      for (int j = 0; j < k; ++j) {
        const double kv = j + 1;
        const int re = ctx->h_stat[4 + j];
        second += re;
        if (ctx->opts.precond)
          prof_work(ctx, FR_KF_APPLY, 8.0 * (double)ctx->ne * ctx->nb * ctx->nb + 24.0 * nd, 2.0 * ctx->nb * nd);
        else
          prof_work(ctx, FR_KF_APPLY, 24.0 * nd, 3.0 * nd);
        prof_work(ctx, FR_KF_JV, 32.0 * nd, jv_flops_per_element(ctx) * (double)ctx->ne + 6.0 * nd);
        // pass 1: dots of j+1 basis vectors and w with w; update reads them and w, writes w
        prof_work(ctx, FR_KF_DOTS, 8.0 * (kv + 1) * nd, 2.0 * (kv + 1) * nd);
        prof_work(ctx, FR_KF_UPDATE, 8.0 * (kv + 2) * nd, 2.0 * kv * nd + 2.0 * nd);
        if (re) {
          prof_work(ctx, FR_KF_DOTS, 8.0 * (kv + 1) * nd, 2.0 * kv * nd);
          prof_work(ctx, FR_KF_UPDATE, 8.0 * (kv + 2) * nd, 2.0 * kv * nd + 2.0 * nd);
        }
      }
      Prof& P = ctx->prof;
      P.skipped[FR_KF_APPLY] += sk;
      P.skipped[FR_KF_JV] += sk;
      P.skipped[FR_KF_DOTS] += 2 * sk + (k - second);
      P.skipped[FR_KF_UPDATE] += 2 * sk + (k - second);
      P.skipped[FR_KF_OTHER] += sk;
    }
    if (!std::isfinite(res) || !std::isfinite(bn)) {
      if (info) *info = loc;
      return set_error(ctx, FR_ERR_NONFINITE, "GMRES residual is not finite");
    }
    if (bn == 0.0) {  // b = 0 and x = 0 on entry
      loc.converged = 1;
      loc.relres = 0.0;
      status = FR_OK;
      break;
    }
    loc.iters += k;
    if (k > 0) ++cycles_iterated;
    loc.relres = res / bn;
    if (res <= target) {
      loc.converged = 1;
      status = FR_OK;
      break;
    }
  }
  loc.restarts = cycles_iterated > 0 ? cycles_iterated - 1 : 0;
  if (info) *info = loc;
  if (status != FR_OK)
    set_error(ctx, FR_ERR_NOT_CONVERGED, "GMRES stopped after %d iterations at relres %.3e",
              loc.iters, loc.relres);
  return status;
}

}  // namespace frk
