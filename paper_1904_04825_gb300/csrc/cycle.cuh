// Restarted GMRES(m) of one linear solve in one launch.
//
// The launches of krylov.cu take seven kernels per Arnoldi iteration, and on a
// small mesh each of them is latency (5 us of host time to launch, 5 to 20 us to
// run).  Here every CTA of a
// resident grid walks through the phases of the same iteration (apply, A z, dot
// products, update, Givens) with a barrier between them (1.3 us at 152 CTAs, 2.2
// us at 608), over all cycles of the solve:
//   * a phase's work items are the blocks of the launch it stands for (vector
//     blocks, apply blocks, element tiles); CTA c of n takes items c, c + n, ...
//     and writes each item's partial sum to the slot that block has, so every sum
//     runs in the same order and the results equal those of the launches bit for
//     bit, whatever n is;
//   * every CTA sums the partials it needs itself after the barrier instead of
//     waiting for a last block; the last CTA also keeps the Hessenberg column and
//     the rotations, while the others start the next apply.
// What an iteration takes at 14,400 unknowns (p = 2, one CTA per SM): apply 6 us,
// A z 11, dot products 5 and their totals 5, update 3, four barriers 7: FP64
// latency and issue, 41 us against 80 by launches.
// The grid is launched cooperatively, so all CTAs are resident; every wait is
// bounded, and a wait that gives up sets *err and ends the CTA.
#pragma once

#include <atomic>

#include "apply_body.cuh"
#include "cycle.h"
#include "krylov_body.cuh"
#include "residual_body.cuh"

namespace frk {
namespace cyc {

constexpr int kColApply = kCycleDots, kColUpdate = kCycleDots + 1, kColU = kCycleDots + 2, kColB = kCycleDots + 3,
              kColX = kCycleDots + 4;  // partial-sum columns beside the dot products'
static_assert(kColX < kMaxVec, "partial columns");

// what a CTA keeps in shared memory beside the phase's buffer
struct Shared {
  double sh[32];
  double tot[kMaxVec + 2];   // totals of the last reduction
  double neg_h[kMaxVec];
  double ys[kMaxVec];
  double eps2[2];
  int flag;                  // of the last barrier: done bit, -1 if it gave up
};

struct Grid {
  unsigned* counter;
  unsigned target, polls;
  int bid, nblk;
  bool ok;
};
// The barrier counter: arrivals times two, which wrap at 2^32 (a solve may take any
// number of barriers; the CTAs are never more than one barrier apart), and in bit 0
// whether the cycle is done (set and cleared by the keeper).
constexpr unsigned kDone = 1u, kArrival = 2u;

// All CTAs of the instance arrive (this one adding `add`, 0 or +-kDone, to the done
// bit), then all see what any of them wrote before.  s.flag: the done bit, which
// is settled at this barrier if the keeper changed it while arriving here or
// earlier.  Returns false when the wait gave up after `polls` looks.
static __device__ __noinline__ bool barrier(Grid& g, Shared& s, unsigned add = 0u) {
  g.target += kArrival * (unsigned)g.nblk;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(g.counter, kArrival + add);
    int flag = -1;
    for (unsigned it = 0; it < g.polls; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(g.counter) : "memory");
      if ((int)((v & ~kDone) - g.target) >= 0) {
        flag = (int)(v & kDone);
        break;
      }
    }
    s.flag = flag;
  }
  __syncthreads();
  g.ok = s.flag >= 0;
  return g.ok;
}

// totals of the columns col .. col + n - 1 over nblk partials into s.tot (all threads)
__device__ __forceinline__ void totals(const Reduce& red, int col, int n, int nblk, Shared& s) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = wid; i < n; i += nw) {
    const double t = sum_partials(red.value(col + i), nblk);
    if (lane == 0) s.tot[i] = t;
  }
  __syncthreads();
}

// partials of ||x||^2 in column col
static __device__ __noinline__ void sumsq_phase(const CycleArgs& a, const double* x, int col, const Grid& g, Shared& s) {
  for (int i = g.bid; i < a.vgrid; i += g.nblk) {
    const double bs = block_sum(sumsq_rows(x, a.n, i, a.vgrid), s.sh);
    if (threadIdx.x == 0) a.red.value(col)[i] = bs;
  }
}

__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The apply of blocks.cu without the staging: z_e = M_e^-1 (sc r_e), r_e *= sc,
// partials of ||z||^2.  Teams of one apply block's threads; a team's row sums run
// over the same KS column ranges in the same order.
template <int NB, typename S, typename A>
__device__ __noinline__ void apply_phase(const CycleArgs& a, double* r, double sc, const Grid& g,
                                            unsigned char* smem) {
  using L = ApplyLayout<NB, S, A>;
  constexpr int KS = L::KS, KP = NB / KS, T = L::THREADS, TEAMS = kCycleThreads / T > 0 ? kCycleThreads / T : 1;
  static_assert(T <= kCycleThreads && TEAMS <= 15, "a team fits the CTA and has a barrier of its own");
  A* base = reinterpret_cast<A*>(smem);
  double* wsum = reinterpret_cast<double*>(smem + (size_t)TEAMS * (2 + KS) * NB * sizeof(A) + 16);
  const int team = threadIdx.x / T, tid = threadIdx.x % T;
  if (team >= TEAMS) return;
  A* rs = base + (size_t)team * (2 + KS) * NB;  // two copies of r, then the partial sums
  A* part = rs + 2 * NB;
  const int i = tid % NB, ks = tid / NB;
  const S* M = reinterpret_cast<const S*>(a.Minv);
  // the keeper, still at its rotations, takes none while others can
  const int workers = g.nblk > 8 ? g.nblk - 1 : g.nblk;
  if (g.bid >= workers) return;
  for (int b = g.bid * TEAMS + team; b < a.agrid; b += workers * TEAMS) {
    double ss = 0.0;
    int buf = 0;
    for (long long e = b; e < a.ne; e += a.agrid, buf ^= 1) {
      A* rb = rs + buf * NB;
      if (ks == 0) {
        const double v = r[e * NB + i] * sc;
        r[e * NB + i] = v;
        rb[i] = (A)v;
      }
      named_barrier(1 + team, T);
      A zz = 0;
      if (ks < KS) {
        const S* Mk = M + e * NB * NB + (size_t)(ks * KP) * NB + i;
        const A* rk = rb + ks * KP;
        A acc0 = 0, acc1 = 0;
#pragma unroll
        for (int k = 0; k < KP; k += 2) {
          acc0 = fma(load_acc(Mk + k * NB), rk[k], acc0);
          if (k + 1 < KP) acc1 = fma(load_acc(Mk + (k + 1) * NB), rk[k + 1], acc1);
        }
        zz = acc0 + acc1;
        if (KS > 1) part[ks * NB + i] = zz;
      }
      if (KS > 1) named_barrier(1 + team, T);
      if (ks == 0) {
        if (KS > 1) {
          zz = part[i];
#pragma unroll
          for (int u = 1; u < KS; ++u) zz += part[u * NB + i];
        }
        const double zi = (double)zz;
        a.z[e * NB + i] = zi;
        ss = fma(zi, zi, ss);
      }
    }
    // the block's sum in the order of block_sum
    ss = warp_sum(ss);
    if ((tid & 31) == 0) wsum[team * (T / 32) + tid / 32] = ss;
    named_barrier(1 + team, T);
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < T / 32; ++w) t += wsum[team * (T / 32) + w];
      a.red.value(kColApply)[b] = t;
    }
    named_barrier(1 + team, T);
  }
}

// x (+)= M^-1 (sum_l y_l V_l), one thread per row
template <int NB, typename S, typename A>
__device__ __noinline__ void solution_phase(const CycleArgs& a, double* x, int k, const double* ys, bool x_zero,
                                               const Grid& g, unsigned char* smem) {
  constexpr int EPC = RowsShape<NB>::EPC;
  A* ts = reinterpret_cast<A*>(smem);
  const S* M = reinterpret_cast<const S*>(a.Minv);
  const int el = threadIdx.x / NB, i = threadIdx.x % NB;
  for (long long e0 = (long long)g.bid * EPC; e0 < a.ne; e0 += (long long)g.nblk * EPC) {
    const long long e = e0 + el;
    const bool act = el < EPC && e < a.ne;
    __syncthreads();
    if (act) {
      double t = 0.0;
      for (int l = 0; l < k; ++l) t = fma(ys[l], a.V[l * a.n + e * NB + i], t);
      ts[el * NB + i] = (A)t;
    }
    __syncthreads();
    if (act) {
      const S* Me = M + e * (long long)NB * NB;
      A acc = 0;
#pragma unroll 16
      for (int kk = 0; kk < NB; ++kk) acc = fma(load_acc(Me + kk * NB + i), ts[el * NB + kk], acc);
      x[e * NB + i] = (x_zero ? 0.0 : x[e * NB + i]) + (double)acc;
    }
  }
}

// out = b - A v, or A v where b is null, with the FD step for ||v||^2 = nv2
template <int P, int TV, int RM>
__device__ __noinline__ void product_phase(const CycleArgs& a, const double* v, const double* b, double* out,
                                              double nU2, double nv2, const Grid& g, Shared& s, unsigned char* smem) {
  using Sm = ResSmem<P, TV>;
  constexpr int TX = Tile<P, TV>::TX, TY = Tile<P, TV>::TY;
  if (threadIdx.x == 0) {
    const EpsArgs ea{&nU2, a.res.eps_rel, a.res.eps_fixed, s.eps2};
    write_eps(ea, nv2);
  }
  __syncthreads();
  const int tiles = ((a.res.nx + TX - 1) / TX) * ((a.res.ny + TY - 1) / TY);
  for (int t = g.bid; t < tiles; t += g.nblk) {
    residual_body<P, 4, TV, RM>(a.res, v, b, s.eps2, out, t, *reinterpret_cast<Sm*>(smem));
    __syncthreads();
  }
}

// partials of <V_i, w>, i < nvec (and of <w, w>), in the columns from 0
static __device__ __noinline__ void dots_phase(const CycleArgs& a, const double* w, int nvec, int total, const Grid& g) {
  for (int q = g.bid; q < a.vgrid; q += g.nblk) dots_partials(a.V, a.n, nvec, w, a.n, total, a.red, q, a.vgrid);
}

// w -= sum_i h_i V_i, partials of the new ||w||^2
static __device__ __noinline__ void update_phase(const CycleArgs& a, double* w, int nvec, const Grid& g, Shared& s) {
  for (int q = g.bid; q < a.vgrid; q += g.nblk) {
    const double bs = block_sum(update_rows(w, a.V, a.n, nvec, s.neg_h, a.n, q, a.vgrid), s.sh);
    if (threadIdx.x == 0) a.red.value(kColUpdate)[q] = bs;
  }
}

// returns whether the cycle is done
static __device__ __noinline__ bool givens_phase(const GmresDev& gd, int j, double nw2) {
  __syncthreads();
  if (threadIdx.x < 32) givens_body(gd, j, &nw2);
  __syncthreads();
  return *(volatile const int*)gd.done != 0;
}

template <int P, int TV, int RM, typename S, typename A>
__device__ __noinline__ void solve(const CycleArgs& a, Grid& g, Shared& s, unsigned char* smem) {
  constexpr int NB = 4 * (P + 1) * (P + 1);
  const GmresDev& gd = a.gd;
  const long long n = a.n;
  const double* b = a.b;
  double* x = a.x;
  const bool keeper = g.bid == g.nblk - 1;  // the CTA that keeps the Hessenberg column
  bool x_zero = a.x_zero != 0;
  int iters = 0, iterated = 0, state = kCycleNotConverged;
  double res = 0.0, target = 0.0, relres = 0.0;
  unsigned done_add = 0u;  // keeper's thread 0: what its next arrival adds
  bool done_set = false;   // ... and whether the done bit is set

  sumsq_phase(a, a.res.U, kColU, g, s);
  sumsq_phase(a, b, kColB, g, s);
  if (!x_zero) sumsq_phase(a, x, kColX, g, s);
  if (!barrier(g, s)) return;
  totals(a.red, kColU, x_zero ? 2 : 3, a.vgrid, s);
  const double nU2 = s.tot[0], nb2 = s.tot[1];
  double nx2 = x_zero ? 0.0 : s.tot[2];
  const double bn = sqrt(nb2);
  target = a.rtol * bn;
  if (nb2 == 0.0) {  // b = 0: the solution is x = 0
    for (long long i = (long long)g.bid * blockDim.x + threadIdx.x; i < n; i += (long long)g.nblk * blockDim.x) x[i] = 0.0;
    state = kCycleConverged;
  } else {
    if (!x_zero && nx2 == 0.0) x_zero = true;
    for (int cycle = 0; cycle <= a.max_restarts; ++cycle) {
      // ---- r = b - A x into V[0] ----
      double nr2 = nb2;
      if (x_zero && cycle == 0) {
        for (int q = g.bid; q < a.vgrid; q += g.nblk)
          for (long long i = (long long)q * blockDim.x + threadIdx.x; i < n; i += (long long)a.vgrid * blockDim.x)
            a.V[i] = b[i];
      } else {
        if (cycle > 0) {
          if (!barrier(g, s)) return;  // x is complete
          sumsq_phase(a, x, kColX, g, s);
          if (!barrier(g, s)) return;
          totals(a.red, kColX, 1, a.vgrid, s);
          nx2 = s.tot[0];
        }
        product_phase<P, TV, RM>(a, x, b, a.V, nU2, nx2, g, s, smem);
        if (!barrier(g, s)) return;
        sumsq_phase(a, a.V, kColX, g, s);
        if (!barrier(g, s)) return;
        totals(a.red, kColX, 1, a.vgrid, s);
        nr2 = s.tot[0];
      }
      const double beta = sqrt(nr2);
      res = beta;
      if (keeper) {
        __syncthreads();
        for (int i = threadIdx.x; i <= a.m; i += blockDim.x) gd.g[i] = i == 0 ? beta : 0.0;
        if (threadIdx.x == 0) {
          *gd.target = target;
          *gd.res = beta;
          *gd.k = 0;
          *gd.done = beta <= target ? 1 : 0;
          gd.invh[0] = beta > 0.0 ? 1.0 / beta : 0.0;
        }
        __syncthreads();
        const bool d = beta <= target;
        done_add = d == done_set ? 0u : (d ? kDone : 0u - kDone);
        done_set = d;
      }
      double sc = beta > 0.0 ? 1.0 / beta : 0.0;
      if (!barrier(g, s, done_add)) return;  // V[0] and the cycle's state
      done_add = 0u;
      const bool fin = s.flag != 0;
      int j = 0;
      for (; j < a.m && !fin; ++j) {
        double* vj = a.V + (size_t)j * n;
        double* w = a.V + (size_t)(j + 1) * n;
        apply_phase<NB, S, A>(a, vj, sc, g, smem);
        if (!barrier(g, s, done_add)) return;
        done_add = 0u;
        if (s.flag) break;  // the iteration before had converged
        totals(a.red, kColApply, 1, a.agrid, s);
        const double nz2 = s.tot[0];
        product_phase<P, TV, RM>(a, a.z, nullptr, w, nU2, nz2, g, s, smem);
        if (!barrier(g, s)) return;
        dots_phase(a, w, j + 1, j + 2, g);
        if (!barrier(g, s)) return;
        totals(a.red, 0, j + 2, a.vgrid, s);
        const double self2 = s.tot[j + 1];
        for (int i = threadIdx.x; i <= j; i += blockDim.x) {
          s.neg_h[i] = -s.tot[i];
          if (keeper) {
            gd.h1[i] = s.tot[i];
            gd.h2[i] = 0.0;
          }
        }
        __syncthreads();
        double nw2;
        for (int pass = 0;; ++pass) {
          update_phase(a, w, j + 1, g, s);
          if (!barrier(g, s)) return;
          totals(a.red, kColUpdate, 1, a.vgrid, s);
          nw2 = s.tot[0];
          if (pass == 1 || !(nw2 < a.eta2 * self2)) break;
          // second Gram-Schmidt pass
          dots_phase(a, w, j + 1, j + 1, g);
          if (!barrier(g, s)) return;
          totals(a.red, 0, j + 1, a.vgrid, s);
          for (int i = threadIdx.x; i <= j; i += blockDim.x) {
            s.neg_h[i] = -s.tot[i];
            if (keeper) gd.h2[i] = s.tot[i];
          }
          __syncthreads();
        }
        if (keeper && givens_phase(gd, j, nw2)) {
          done_add = kDone;
          done_set = true;
        }
        const double hn = sqrt(nw2);
        sc = hn > 0.0 ? 1.0 / hn : 0.0;
      }
      if (j == a.m) {  // the last column is the keeper's: everyone waits for it
        if (!barrier(g, s, done_add)) return;
        done_add = 0u;
      }
      // ---- x += M^-1 V y ----
      const int k = *(volatile const int*)gd.k;
      res = *(volatile const double*)gd.res;
      if (k > 0) {
        backsub(gd, k, reinterpret_cast<double*>(smem), s.ys);
        solution_phase<NB, S, A>(a, x, k, s.ys, x_zero && cycle == 0, g, smem);
      }
      if (!isfinite(res) || !isfinite(bn)) {  // the cycles before this one are reported
        state = kCycleNonFinite;
        if (k > 0) ++iterated;
        break;
      }
      iters += k;
      if (k > 0) ++iterated;
      relres = res / bn;
      if (res <= target) {
        state = kCycleConverged;
        break;
      }
    }
    if (x_zero && iterated == 0)  // no iteration: x = 0 all the same
      for (long long i = (long long)g.bid * blockDim.x + threadIdx.x; i < n; i += (long long)g.nblk * blockDim.x) x[i] = 0.0;
  }
  if (keeper && threadIdx.x == 0) {
    CycleStatus* st = a.status;
    st->iters = iters;
    st->restarts = iterated > 0 ? iterated - 1 : 0;
    st->state = state;
    st->relres = relres;
  }
}

template <int RM, typename S, typename A>
__device__ __forceinline__ void run(const CycleArgs& a, int bid, int nblk, Shared& s, unsigned char* smem) {
  Grid g{a.bar, 0u, a.polls, bid, nblk, true};
  switch (a.p * 2 + (a.small_tile ? 1 : 0)) {
    case 4: solve<2, 0, RM, S, A>(a, g, s, smem); break;
    case 5: solve<2, 2, RM, S, A>(a, g, s, smem); break;
    case 6: solve<3, 0, RM, S, A>(a, g, s, smem); break;
    case 7: solve<3, 2, RM, S, A>(a, g, s, smem); break;
    case 8: solve<4, 0, RM, S, A>(a, g, s, smem); break;
    case 9: solve<4, 2, RM, S, A>(a, g, s, smem); break;
  }
  // the last CTA to leave sets the counter back for the next launch and passes the
  // context's flag on (after a wait that gave up the host clears the counter)
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!g.ok) atomicExch(a.err, 1);
    __threadfence();  // the flag before the arrival
    const unsigned t = atomicAdd(a.bar, kArrival) + kArrival;
    if ((t & ~kDone) == g.target + kArrival * (unsigned)nblk) {
      __threadfence();
      a.status->err = *(volatile const int*)a.err;
      atomicExch(a.bar, 0u);
    }
  }
}

template <int RM, typename S, typename A>
__global__ void __launch_bounds__(kCycleThreads, kCyclePerSm) k_cycle(const __grid_constant__ CycleArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ Shared s;
  run<RM, S, A>(a, blockIdx.x, gridDim.x, s, smem);
}

constexpr size_t max_of(size_t a, size_t b) { return a > b ? a : b; }
template <int P, typename S, typename A>
constexpr size_t smem_of() {
  constexpr int NB = 4 * (P + 1) * (P + 1);
  using L = ApplyLayout<NB, S, A>;
  constexpr size_t teams = kCycleThreads / L::THREADS > 0 ? kCycleThreads / L::THREADS : 1;
  return max_of(max_of(sizeof(ResSmem<P, 0>), sizeof(ResSmem<P, 2>)),
                max_of(teams * (2 + L::KS) * NB * sizeof(A) + 16 + 64 * sizeof(double),
                       max_of(kTriangle * sizeof(double), (size_t)RowsShape<NB>::EPC * NB * sizeof(A))));
}
template <typename S, typename A>
constexpr size_t cycle_smem() {
  return max_of(smem_of<2, S, A>(), max_of(smem_of<3, S, A>(), smem_of<4, S, A>()));
}

template <typename S, typename A>
const void* kernel_of(int riemann) {
  return riemann ? (const void*)k_cycle<1, S, A> : (const void*)k_cycle<0, S, A>;
}

template <typename S, typename A>
int launch(const CycleArgs& a, int nblocks, int riemann, cudaStream_t s) {
  count_launch();
  void* args[] = {const_cast<CycleArgs*>(&a)};
  return cudaLaunchCooperativeKernel(kernel_of<S, A>(riemann), dim3(nblocks), dim3(kCycleThreads), args,
                                     cycle_smem<S, A>(), s) == cudaSuccess
             ? FR_OK
             : FR_ERR_CUDA;
}

// resident CTAs per SM, found once per device (with the shared-memory attribute) by
// whichever threads ask first; they find the same
template <typename S, typename A>
int resident(int riemann, int device) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices][2];  // one more than the number; 0: not yet known
  std::atomic<int>* slot = device >= 0 && device < kDevices ? &known[device][riemann] : nullptr;
  int o = slot ? slot->load(std::memory_order_relaxed) - 1 : -1;
  if (o >= 0) return o;
  const void* f = kernel_of<S, A>(riemann);
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cycle_smem<S, A>()) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, f, kCycleThreads, cycle_smem<S, A>()) != cudaSuccess) {
    (void)cudaGetLastError();
    o = 0;
  }
  if (slot) slot->store(o + 1, std::memory_order_relaxed);
  return o;
}

}  // namespace cyc
}  // namespace frk
