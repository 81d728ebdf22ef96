// Arguments and entry points of the GMRES solve in one launch (cycle.cuh).
#pragma once

#include "residual_body.cuh"

namespace frk {

constexpr int kCycleThreads = 256;         // the vector kernels' block size, whose blocks are the work items
constexpr int kCyclePerSm = 2;             // resident CTAs per SM the kernel is compiled for
constexpr int kCycleDots = kMaxVec - 5;    // columns of partial sums for dot products; five more follow
static_assert(kCycleThreads == kThreads, "a work item is one block of the vector kernels");

enum { kCycleConverged = 0, kCycleNotConverged = 1, kCycleNonFinite = 2 };
// how a solve ended
struct CycleStatus {
  int iters, restarts, state;
  int err;                 // the context's flag as the last CTA left; 1 (the host's) if none saw itself as the last
  double relres;
};

// One linear solve A x = b of a 2D Euler context.
struct CycleArgs {
  ResArgs res;             // U, R0, shift, mesh, tables
  int p, small_tile;       // degree; residual tile shape 2 instead of 0
  const void* Minv;
  double* V;
  double* z;
  long long n, ne;
  const double* b;
  double* x;
  Reduce red;
  GmresDev gd;
  double eta2, rtol;
  int m, max_restarts, vgrid, agrid;  // blocks of the vector kernels and of the apply
  int x_zero;              // x is zero on entry (and need not be filled)
  unsigned* bar;           // the grid barriers' counter, zero at the launch
  unsigned polls;          // limit of every wait at a grid barrier
  int* err;                // set when one gave up
  CycleStatus* status;     // pinned host memory
};

// residual.cu
ResArgs residual_args(fr_ctx* ctx, const double* U, const double* R0, double shift);
bool residual_small_tile(const fr_ctx* ctx);

// by the block precision: the launch, and the resident CTAs per SM (0: cannot run)
#define FRK_CYCLE_ENTRY(name)                                                          \
  int launch_cycle_##name(const CycleArgs& a, int nblocks, int riemann, cudaStream_t s); \
  int resident_cycle_##name(int riemann, int device);
FRK_CYCLE_ENTRY(f64)
FRK_CYCLE_ENTRY(f32)
FRK_CYCLE_ENTRY(bf16)
#undef FRK_CYCLE_ENTRY

// whether a solve of restart length m runs as one launch (it then writes x whole
// where the guess is zero; the separate launches add to the zeros they are given);
// the context's arguments; the grid
bool solves_in_one_launch(const fr_ctx* ctx, int m);
int fill_cycle_args(fr_ctx* ctx, const double* U, const double* R0, double shift, double rtol, int m, int max_restarts,
                    CycleArgs* a);
int launch_cycle(int prec, const CycleArgs& a, int nblocks, int riemann, cudaStream_t s);
// one solve in one launch on the stream; its status lies in ctx->h_cyc when it is done
int launch_solve(fr_ctx* ctx, const double* U, const double* R0, double shift, const double* b, double* x, int m,
                 double rtol, int max_restarts, bool x_is_zero, cudaStream_t s);
// CTAs of a solve
int cycle_grid(const fr_ctx* ctx);

}  // namespace frk
