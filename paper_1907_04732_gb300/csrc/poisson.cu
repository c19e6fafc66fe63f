// Poisson solve of the LBE step (Sec. "Imposing conducting boundary
// conditions"): find phi on fluid nodes such that
//     lap_mod(phi)(r) + 4 pi l_B rho_el(r) = 0,
// where lap_mod is Eq. DiscreteLaplacianModif (every fluid-solid link
// doubled) and solid nodes hold their electrode potential.  The paper relaxes
// with Eq. SOR and keeps the converged potential; here the same fixed point is
// reached by iterative refinement:
//
//   round:  res = 4 pi l_B rho_el + lap_mod(phi)      (FP64 in the FP64 form;
//           in the FP32 form lap_mod of the fixed-point potential summed
//           exactly in integers, the sum added to the charge term in
//           float-float arithmetic)
//           stop when max_r |res(r)|/diag(r) <= poisson_tol
//           solve A e = res approximately by preconditioned conjugate
//           gradients with the multigrid V-cycle of mg.cu, in the form's
//           precision (Jacobi where a lattice has no hierarchy)
//           phi += e                (FP64; FP32 form: e rounded to the
//                                    fixed-point unit, an integer add)
//
// Each step starts from the extrapolation in time of the previous solutions
// (fp32::extrapolate_node, fp32::extrapolate_fx).  The CG is the Chronopoulos-Gear variant: both
// inner products of an iteration come from one reduction phase, so an
// iteration is the preconditioner, the stencil with the dot products (k_cg_b,
// whose last block runs the scalar recurrence) and the vector update with the
// stopping test (k_cg_a).  Up to kOneNodes nodes the whole solve is one
// cooperative kernel (k_solve_one).  Beyond, or with Jacobi sweeps on the
// coarsest level, it is one CUDA graph: a device-side `while` over refinement
// rounds containing a `while` over CG iterations; kernels set the loop
// conditions, bounded by the round limit and poisson_max_iter.  Where
// conditional graph nodes are not available the same kernels run from a host
// loop that polls the device.
//
// Reductions are deterministic: each block reduces in a fixed tree order and
// writes one partial; a single block sums the partials in block order.
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "solve_device.cuh"
#include "vcycle.cuh"

namespace lbe {

namespace {

constexpr int kMaxOuter = 24;  // refinement rounds per solve
constexpr int kChunk = 16;     // fallback: iterations between host polls

enum { S_RU = 0, S_WU = 1 };

// block-wide sum or max in a fixed order; result valid in thread 0.  The
// FP32 kernels reduce in FP32 within the block (FP64 is slow on this GPU);
// block partials are stored and combined in FP64.
template <bool MAX, typename V = double>
__device__ __forceinline__ V block_reduce(V v) {
  __shared__ V sh[kBlock / 32];
  const int t = flat_tid(), lane = t & 31, wid = t >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const V u = __shfl_down_sync(0xffffffffu, v, o);
    v = MAX ? fmax(v, u) : v + u;
  }
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  V out = 0;
  if (t == 0) {
    out = sh[0];
    for (int w = 1; w < kBlock / 32; ++w) out = MAX ? fmax(out, sh[w]) : out + sh[w];
  }
  return out;
}

__device__ __forceinline__ void set_cond(cudaGraphConditionalHandle h, int use, unsigned v) {
  if (use) cudaGraphSetConditional(h, v);
}

// Last-block-done: after a block has written its partials it takes a ticket;
// the block that takes the last ticket sees every partial (each block fenced
// its writes before its ticket) and finishes the reduction.  No block waits.
__device__ __forceinline__ bool last_block(PoissonCtl *c, int nblk) {
  __shared__ int last;
  __syncthreads();
  if (flat_tid() == 0) {
    __threadfence();
    last = atomicAdd(&c->arrive, 1) == nblk - 1;
  }
  __syncthreads();
  return last;
}

// two sums over the block in one pass (the order of block_reduce for each
// value, with one pair of barriers); results valid in thread 0
template <typename V>
__device__ __forceinline__ void block_reduce2(V &a, V &b) {
  __shared__ V sh[2][kBlock / 32];
  const int t = flat_tid(), lane = t & 31, wid = t >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const V ua = __shfl_down_sync(0xffffffffu, a, o), ub = __shfl_down_sync(0xffffffffu, b, o);
    a += ua;
    b += ub;
  }
  __syncthreads();
  if (lane == 0) {
    sh[0][wid] = a;
    sh[1][wid] = b;
  }
  __syncthreads();
  if (t == 0) {
    a = sh[0][0];
    b = sh[1][0];
    for (int w = 1; w < kBlock / 32; ++w) {
      a += sh[0][w];
      b += sh[1][w];
    }
  }
}

// sums of the partials in block order (every thread of the block calls).
// A thread's partials of the first kSolveBlocks blocks are loaded before any is
// added (one L2 latency instead of one per stride of the block), then summed in
// the same order; those of further blocks (the stencil has 2048 on the 256^3
// lattice) follow one stride after another.
__device__ __forceinline__ void reduce_partials(const double *part, int nblk, double *ru, double *wu) {
  constexpr int kPer = (kSolveBlocks + kBlock - 1) / kBlock;
  double pa[kPer], pb[kPer];
  const int t = flat_tid();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int i = t + k * kBlock;
    const bool in = i < nblk;
    pa[k] = in ? __ldcg(part + S_RU * nblk + i) : 0.0;
    pb[k] = in ? __ldcg(part + S_WU * nblk + i) : 0.0;
  }
  double a = 0.0, b = 0.0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (t + k * kBlock < nblk) {
      a += pa[k];
      b += pb[k];
    }
  }
  for (int i = t + kPer * kBlock; i < nblk; i += kBlock) {
    a += __ldcg(part + S_RU * nblk + i);
    b += __ldcg(part + S_WU * nblk + i);
  }
  block_reduce2(a, b);
  *ru = a;
  *wu = b;
}

// outer test of a refinement round (thread 0 of the last block of k_res):
// converged, out of rounds or out of iterations?  A round that did not
// halve the residual means the tolerance lies below what the arithmetic
// resolves: the solve stops there (LBE_ERR_NOCONVERGE) instead of repeating
// rounds that cannot help.
__device__ void outer_check(PoissonCtl *c, double m, double tol, int maxit, cudaGraphConditionalHandle hout,
                            cudaGraphConditionalHandle hin, int use_cond) {
  const double prev = c->res;
  c->res = m;
  int done = 0;
  if (m <= tol || c->status) {  // converged, or the round's CG failed
    done = 1;
  } else if (!(m == m) || m > 1e300) {
    done = 1;
    c->status = LBE_ERR_NONFINITE;
  } else if (c->rounds >= kMaxOuter || c->solve_iters >= maxit || (c->rounds >= 1 && m > 0.5 * prev)) {
    done = 1;
    c->status = LBE_ERR_NOCONVERGE;
  }
  c->outer_done = done;
  c->inner_done = done;  // nothing more of the round runs once converged
  c->round_iters = 0;
  c->rounds += 1;
  c->total_rounds += 1;
  set_cond(hout, use_cond, done ? 0u : 1u);
  set_cond(hin, use_cond, done ? 0u : 1u);
}

// scalar recurrence of the Chronopoulos-Gear CG (thread 0 of the last block
// of k_cg_b): step lengths of the update that follows.  A breakdown (the
// correction is converged to rounding, or a zero residual) ends the inner
// solve without an update.
__device__ void cg_scalars(PoissonCtl *c, double gam, double del, cudaGraphConditionalHandle hin, int use_cond) {
  int done = 0;
  if (c->round_iters == 0) {
    c->beta = 0.0;
    c->alpha = gam / del;
    c->gamma = gam;
    if (!(del > 0.0) || !(gam > 0.0)) done = 1;
  } else if (!(del == del)) {
    done = 1;
    c->status = LBE_ERR_NONFINITE;
  } else {
    const double beta = gam / c->gamma;
    const double den = del - beta * gam / c->alpha;
    if (!(den > 0.0) || !(gam > 0.0)) {
      done = 1;
    } else {
      c->beta = beta;
      c->alpha = gam / den;
      c->gamma = gam;
    }
  }
  if (done) {
    c->inner_done = 1;
    set_cond(hin, use_cond, 0u);
  }
}

// inner stopping test (relative reduction eta of the round's starting
// residual) on the updated residual; thread 0 of the last block of k_cg_a
__device__ void cg_test(PoissonCtl *c, double mx, double eta, double tol_abs, int maxit,
                        cudaGraphConditionalHandle hin, int use_cond) {
  int done = 0;
  c->round_iters += 1;
  c->solve_iters += 1;
  c->total_iters += 1;
  if (mx <= fmax(eta * c->res, tol_abs)) {
    done = 1;
  } else if (!(mx == mx) || mx > 1e300) {
    done = 1;
    c->status = LBE_ERR_NONFINITE;
  } else if (c->solve_iters >= maxit) {
    done = 1;
  }
  c->inner_done = done;
  set_cond(hin, use_cond, done ? 0u : 1u);
}

// ---------------------------------------------------------------------------
// start of a solve: fold the previous solve into the sticky fields, reset
__device__ __forceinline__ void solve_reset(PoissonCtl *c) {
  if (c->status && !c->sticky_status) c->sticky_status = c->status;
  if (c->solve_iters > c->max_solve_iters) c->max_solve_iters = c->solve_iters;
  c->outer_done = 0;
  c->inner_done = 0;
  c->rounds = 0;
  c->status = 0;
  c->solve_iters = 0;
  c->solves += 1;
}
__global__ void k_solve_reset(PoissonCtl *c) { solve_reset(c); }

template <typename T, int MODE>
__global__ void __launch_bounds__(kBlock) k_res(const ResArgs A, T *__restrict__ r, T *__restrict__ uj) {
  constexpr bool RHS = kRhs<MODE>;
  float mx = 0.f, mb = 0.f;
  Column c;
  if (column_of(A.cols, c)) res_column<T, MODE>(A, c, r, uj, mx, mb);
  mx = block_reduce<true, float>(mx);
  if (RHS) mb = block_reduce<true, float>(mb);
  if (flat_tid() == 0) {
    PoissonCtl *ctl = A.c;
    atomicMax(&ctl->max_bits, (unsigned long long)__double_as_longlong((double)mx));
    if (RHS) atomicMax(&ctl->ref_bits, (unsigned long long)__double_as_longlong((double)mb));
    __threadfence();
    if (atomicAdd(&ctl->arrive, 1) == A.nblk - 1) {
      const double m = __longlong_as_double((long long)atomicExch(&ctl->max_bits, 0ULL));
      double ref = 0.0;
      if (RHS) {
        ref = __longlong_as_double((long long)atomicExch(&ctl->ref_bits, 0ULL));
        ctl->ref = ref;
      }
      ctl->arrive = 0;
      outer_check(ctl, m, RHS ? fmax(A.tol, A.tol_rel * ref) : A.tol, A.maxit, A.hout, A.hin, A.use_cond);
    }
  }
}

// stencil + dot products: w = A u; partials (r,u), (w,u); the last block
// runs the scalar recurrence.  Marched (march.cuh); u is zero on solid nodes
// and w is set to zero there, so that the update needs no mask.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_cg_b(const Cols C, const uint8_t *__restrict__ code,
                                                 const T *__restrict__ u, const T *__restrict__ r,
                                                 T *__restrict__ w, double *__restrict__ part, int nblk,
                                                 PoissonCtl *c, cudaGraphConditionalHandle hin, int use_cond) {
  if (!use_cond && c->inner_done) return;  // the graph's loop has ended by then
  T ru = 0, wu = 0;
  Column col;
  if (column_of(C, col)) cg_b_column(C, col, code, u, r, w, ru, wu);
  block_reduce2(ru, wu);
  if (flat_tid() == 0) {
    part[S_RU * nblk + flat_bid()] = (double)ru;
    part[S_WU * nblk + flat_bid()] = (double)wu;
  }
  if (!last_block(c, nblk)) return;
  double gam, del;
  reduce_partials(part, nblk, &gam, &del);
  if (flat_tid() == 0) {
    c->arrive = 0;
    cg_scalars(c, gam, del, hin, use_cond);
  }
}

// VEC consecutive values as one load or store (16 bytes; the codes VEC bytes)
template <typename T, int VEC>
struct alignas(sizeof(T) * VEC) Pack {
  T v[VEC];
};

// vector update: p = u + beta p, s = w + beta s, x += alpha p,
// r -= alpha s, uj = r/diag; the last block runs the stopping test on
// max |r|/diag, so that the loop ends here.  (With the test in the stencil
// kernel, the round's last V-cycle and stencil served only to carry it: on
// the 64x64x256 electro-osmosis lattice, tolerance 1e-13, the solve took
// 388 us per step instead of 333.)  A round's first update starts x, p and s
// instead of reading zeros that the residual kernel would have to write.
// Every vector is zero on solid nodes, so no node waits for its mask.
template <typename T, int VEC>
__device__ __forceinline__ T cg_a_nodes(long long N, long long k0, long long dk, const uint8_t *code, T *x, T *r,
                                        const T *u, T *uj, const T *w, T *p, T *s, T alpha, T beta, bool first) {
  using PT = Pack<T, VEC>;
  using PC = Pack<uint8_t, VEC>;
  T mx = 0;
  const long long n = N / VEC;
  for (long long k = k0; k < n; k += dk) {
    const PT uv = ((const PT *)u)[k], wv = ((const PT *)w)[k];
    PT rv = ((PT *)r)[k];
    const PC cv = ((const PC *)code)[k];
    PT pv = uv, sv = wv, xv, jv;
    if (first) {
#pragma unroll
      for (int e = 0; e < VEC; ++e) xv.v[e] = alpha * uv.v[e];
    } else {
      const PT p0 = ((PT *)p)[k], s0 = ((PT *)s)[k];
      xv = ((PT *)x)[k];
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        pv.v[e] = uv.v[e] + beta * p0.v[e];
        sv.v[e] = wv.v[e] + beta * s0.v[e];
        xv.v[e] += alpha * pv.v[e];
      }
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      rv.v[e] -= alpha * sv.v[e];
      const T dinv = inv_diag<T>(cv.v[e]);
      jv.v[e] = rv.v[e] * dinv;
      mx = fmax(mx, finite_or_inf(fabs(rv.v[e]) * dinv));
    }
    ((PT *)p)[k] = pv;
    ((PT *)s)[k] = sv;
    ((PT *)x)[k] = xv;
    ((PT *)r)[k] = rv;
    ((PT *)uj)[k] = jv;
  }
  return mx;
}
template <typename T, int VEC>
__global__ void __launch_bounds__(kBlock) k_cg_a(long long N, const uint8_t *__restrict__ code, T *__restrict__ x,
                                                 T *__restrict__ r, const T *u, T *uj,
                                                 const T *__restrict__ w, T *__restrict__ p, T *__restrict__ s,
                                                 int nblk, PoissonCtl *c, double eta, double tol_abs, int maxit,
                                                 cudaGraphConditionalHandle hin, int use_cond) {
  if (c->inner_done) return;  // a breakdown in this iteration
  const T mx = cg_a_nodes<T, VEC>(N, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x,
                                  code, x, r, u, uj, w, p, s, (T)c->alpha, (T)c->beta, c->round_iters == 0);
  // a maximum does not depend on the order: the blocks combine theirs in one
  // word (the bits of a non-negative double order as an integer), and the
  // last ticket's thread has no partials to read
  const T v = block_reduce<true, T>(mx);
  if (flat_tid() == 0) {
    atomicMax(&c->max_bits, (unsigned long long)__double_as_longlong((double)v));
    __threadfence();
    if (atomicAdd(&c->arrive, 1) == nblk - 1) {
      const double m = __longlong_as_double((long long)atomicExch(&c->max_bits, 0ULL));
      c->arrive = 0;
      cg_test(c, m, eta, tol_abs, maxit, hin, use_cond);
    }
  }
}

// warm start of a step's solve on fluid nodes (fp32::extrapolate_node); the
// FP32 form with flow does this inside the advection kernel instead
__global__ void k_extrapolate(const Geo g, int zpt, const uint32_t *__restrict__ mask, double *__restrict__ phi,
                              double *__restrict__ prev, float *__restrict__ phi32, float *__restrict__ phi_lo,
                              int history) {
  for (int kz = 0; kz < zpt; ++kz) {
    int X, Y, Z;
    long long i;
    if (!node_of(g, zpt, kz, X, Y, Z, i)) continue;
    if (mask[i] & kFluidBit) fp32::extrapolate_node(g.N, i, phi, prev, phi32, phi_lo, history);
  }
}

// FP32 form: the fixed-point potential += e (rounded to the fixed-point
// unit) and its float copy; |phi| reaching kPhiMax raises range flag 4.  e is
// zero on solid nodes, which keep their values.
__device__ __forceinline__ void correct_fx_nodes(long long N, long long k0, long long dk, const float *e, int64_t *phifx,
                                                 float *phi32, int *flag) {
  constexpr float kMaxFx = (float)(kPhiMax * 281474976710656.0);  // kPhiMax 2^kPhiFixBits
  bool over = false;
#pragma unroll 4
  for (long long i = k0; i < N; i += dk) {
    const float d = __fmul_rn(e[i], 281474976710656.0f);  // e 2^kPhiFixBits, exact
    const bool bad = !(fabsf(d) < kMaxFx);  // also NaN
    const long long v = phifx[i] + (bad ? 0LL : fp32::f2ll_rn(d));
    over |= bad || !(fabsf(fp32::ll2f(v)) < kMaxFx);
    phifx[i] = v;
    phi32[i] = fp32::fx_to_f(v);
  }
  if (over) atomicOr(flag, 4);
}
__global__ void __launch_bounds__(kBlock) k_correct_fx(long long N, const float *__restrict__ e,
                                                       int64_t *__restrict__ phifx, float *__restrict__ phi32,
                                                       int *__restrict__ flag, const PoissonCtl *__restrict__ c) {
  if (c->outer_done || c->round_iters == 0) return;  // converged, or no update in this round
  correct_fx_nodes(N, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, e, phifx,
                   phi32, flag);
}

// FP32 form without flow (no advection kernel to carry it): the warm start
// on the fixed-point potential
__global__ void k_extrapolate_fx(const Geo g, int zpt, const uint32_t *__restrict__ mask, int64_t *__restrict__ phifx,
                                 int64_t *__restrict__ prev, float *__restrict__ phi32, int history) {
  for (int kz = 0; kz < zpt; ++kz) {
    int X, Y, Z;
    long long i;
    if (!node_of(g, zpt, kz, X, Y, Z, i)) continue;
    if (mask[i] & kFluidBit) fp32::extrapolate_fx(g.N, i, phifx, prev, phi32, history);
  }
}

// phi64 += e (zero on solid nodes); with phi32 given its float split follows
// (the FP64 form, and the linear solves' FP64 iterates)
template <typename T>
__device__ __forceinline__ void correct_nodes(long long N, long long k0, long long dk, const T *e, double *phi, float *phi32,
                                              float *phi_lo) {
#pragma unroll 4
  for (long long i = k0; i < N; i += dk) {
    double v = phi[i];
    if (e) {
      v += (double)e[i];
      phi[i] = v;
    }
    if (phi32) {
      const float hi = (float)v;
      phi32[i] = hi;
      if (phi_lo) phi_lo[i] = (float)(v - (double)hi);
    }
  }
}
template <typename T>
__global__ void __launch_bounds__(kBlock) k_correct(long long N, const T *__restrict__ e, double *__restrict__ phi,
                                                    float *__restrict__ phi32, float *__restrict__ phi_lo,
                                                    const PoissonCtl *__restrict__ c) {
  if (c && (c->outer_done || c->round_iters == 0)) return;  // converged, or no update in this round
  correct_nodes(N, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, e, phi, phi32,
                phi_lo);
}

// ---------------------------------------------------------------------------
// The whole solve as one cooperative kernel, for lattices whose kernels are
// too short to fill the GPU.  There an iteration of the graph (five to nine
// kernels and a conditional node) is launch, ramp and drain: 35-40 us per
// iteration on a 32x32x16 or a 128x128x4 lattice, 23-26 us here.  The same
// bodies run as phases of resident blocks with a barrier of the grid between
// them; each block keeps the control block in shared memory and runs the
// scalar recurrence and the tests itself on the same partials, in the same
// order.  What is left of a small lattice's phase is the latency of the
// barrier (a release, a poll, L1 refilled) and of two dependent L2 reads.
struct GridBar {
  unsigned count;
  unsigned exits;  // blocks that left; kDeadExit more for each whose wait ran out
  int dead;
};
constexpr unsigned kDeadExit = 1u << 16;
// polls of a wait, some seconds: one that long never ends.  LBE_SOLVE_SPINS sets
// another limit (0: a wait that is not over at its first poll runs out).
constexpr int kSpinLimit = 1 << 23;

// All blocks of the (cooperative, hence co-resident) grid have arrived and
// their writes are visible; false when the wait ran out, in every thread of
// the block (the caller returns, other blocks see `dead` and do the same).
__device__ __forceinline__ bool grid_sync(GridBar *b, int limit, unsigned &target) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    target += gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&b->count) : "memory");
    unsigned v;
    int good = 1;
    for (int spins = 0;; ++spins) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&b->count) : "memory");
      if ((int)(v - target) >= 0) break;
      if (spins >= limit || ((spins & 1023) == 1023 && *(volatile int *)&b->dead)) {
        *(volatile int *)&b->dead = 1;
        good = 0;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok;
}

template <typename T>
struct OneArgs {
  ResArgs R;
  mgd::VCycleArgs<T> V;
  T *r, *u, *uj, *w, *x, *p, *s;
  double *phi;
  float *phi32, *phi_lo;
  int64_t *phifx;
  int *flag;
  double *part;  // [3][blocks]: (r,u), (w,u), maxima
  GridBar *bar;
  int spins;     // limit of a wait
  long long N;
  double eta, tol_inner;
  int cbl;         // log2 of the columns of a block
  int gx, blocks;  // column blocks, and all (column, chunk) blocks
  int vec;         // the update takes 16 bytes at a time
};

// Lattices up to this size take the single-kernel solve.  Both paths, ms per
// solve (one kernel / graph): FP32 16x16x64 0.046 / 0.082, 128x128x4 driven
// coax 0.316 / 0.454, 61x47x53 electrodes 0.278 / 0.351, 64x64x256 0.244 /
// 0.276, porous 128x128x64 0.452 / 0.487; 128x128x128 0.395 / 0.380 and
// 128x128x256 0.751 / 0.671, where a kernel of its own keeps more warps in
// flight.  FP64 4x4x64 0.064 / 0.105, 128x128x4 coax 0.368 / 0.462, 64x64x256
// 0.915 / 0.980.
constexpr long long kOneNodes = 3 << 19;
// Resident blocks: at most so many per SM (FP32 at 64x64x256 with 1, 2, 3:
// 0.382, 0.274, 0.251 ms; FP64 at 128x128x4 0.368 with one, 0.456 with two,
// every block repeating the FP64 reductions), as many as the stencils have
// blocks of columns, and one per SM where only the matrix's rows are more.
template <typename T>
constexpr int kOnePerSM = sizeof(T) == 4 ? 3 : 1;
constexpr int kOneBlocks = 608;  // room for the partials
static_assert(kOneBlocks < (int)kDeadExit, "exits are counted in the low half of the word");
enum { ONE_RU = 0, ONE_WU = 1, ONE_MAX = 2, ONE_REF = 1 };

// Two values of every block combined in block order; valid in thread 0.  All
// threads fetch them (one L2 latency), one warp adds each (an FP64
// instruction holds the narrow pipe for 16 cycles).
__device__ __forceinline__ void grid_sums(const double *a_, const double *b_, double &a, double &b) {
  __shared__ double sv[2][kOneBlocks], sum_b;
  const int G = gridDim.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < (kOneBlocks + kBlock - 1) / kBlock; ++k) {
    const int i = threadIdx.x + k * kBlock;
    if (i < G) {
      sv[0][i] = __ldcg(a_ + i);
      sv[1][i] = __ldcg(b_ + i);
    }
  }
  __syncthreads();
  double v = 0.0;
  if (w < 2) {
    for (int i = lane; i < G; i += 32) v += sv[w][i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (w == 1 && lane == 0) sum_b = v;
  }
  __syncthreads();
  a = v;
  b = sum_b;
}
// maxima of the blocks' (non-negative) values, whose bits order as integers
__device__ __forceinline__ double grid_max(const double *a_) {
  const long long *a = reinterpret_cast<const long long *>(a_);
  __shared__ long long sm[kBlock / 32];
  const int G = gridDim.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long v = 0;
#pragma unroll
  for (int k = 0; k < (kOneBlocks + kBlock - 1) / kBlock; ++k) {
    const int i = threadIdx.x + k * kBlock;
    if (i < G) v = max(v, __ldcg(a + i));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_down_sync(0xffffffffu, v, o));
  if (lane == 0) sm[w] = v;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 1; k < kBlock / 32; ++k) v = max(v, sm[k]);
  return __longlong_as_double(v);
}

// u = M r; every phase but the last ends in a barrier.  false: a wait ran out
template <typename T>
__device__ __forceinline__ bool one_vcycle(const OneArgs<T> &S, unsigned &target) {
  using namespace mgd;
  const VCycleArgs<T> &V = S.V;
  const int G = gridDim.x, b0 = blockIdx.x, warp = threadIdx.x >> 5;
  for (int b = b0; b < V.g0x * V.g0y * V.g0z; b += G) {
    const int bx = b % V.g0x, t = b / V.g0x;
    restrict0_block(S.R.cols, S.R.code, S.r, S.uj, V.lv[1], V.W[1], V.r[1], V.z[1], V.M, bx, t % V.g0y, t / V.g0y);
  }
  if (!grid_sync(S.bar, S.spins, target)) return false;
  for (int l = 1; l < V.ld; ++l) {
    for (int b = b0; b < V.rx[l] * V.ry[l] * V.rz[l]; b += G) {
      const int bx = b % V.rx[l], t = b / V.rx[l];
      restrict_block(V.lv[l], V.A[l], V.r[l], V.z[l], V.lv[l + 1], V.W[l + 1], V.r[l + 1], V.z[l + 1], V.txl[l], bx,
                     t % V.ry[l], t / V.ry[l]);
    }
    if (!grid_sync(S.bar, S.spins, target)) return false;
  }
  for (int row = b0 * (kBlock / 32) + warp; row < V.ndense; row += G * (kBlock / 32)) {
    if (V.stride) dense_row(row, V.stride, V.mat, V.r[V.ld], V.e[V.ld]);
    else inverse_row(row, V.ndense, V.mat, V.r[V.ld], V.e[V.ld]);
  }
  if (!grid_sync(S.bar, S.spins, target)) return false;
  for (int l = V.ld - 1; l >= 1; --l) {
    for (int i = b0 * kBlock + threadIdx.x; i < V.lv[l].N; i += G * kBlock) {
      int X, Y, Z;
      level_coords(V.lv[l], i, X, Y, Z);
      V.e[l][i] = post_value_w<T>(V.lv[l], V.A[l], V.W[l][i], V.r[l], V.z[l], V.lv[l + 1], V.e[l + 1], X, Y, Z);
    }
    if (!grid_sync(S.bar, S.spins, target)) return false;
  }
  for (int b = b0; b < S.blocks; b += G) {
    Column c;
    if (block_column(S.R.cols, S.cbl, S.gx, b, (int)threadIdx.x, c))
      post0_column(S.R.cols, c, S.R.code, S.R.mask, S.r, S.uj, V.lv[1], V.e[1], S.u);
  }
  return true;
}

// false: a wait ran out
template <typename T, int MODE>
__device__ __forceinline__ bool one_solve(const OneArgs<T> &S, PoissonCtl *sc, unsigned &target) {
  const int G = gridDim.x, b0 = blockIdx.x, t = threadIdx.x;
  const long long k0 = (long long)b0 * kBlock + t, dk = (long long)G * kBlock;
  double m0, m1;
  for (;;) {
    float mx = 0.f, mb = 0.f;
    for (int b = b0; b < S.blocks; b += G) {
      Column c;
      if (block_column(S.R.cols, S.cbl, S.gx, b, t, c))
        res_column<T, MODE>(S.R, c, S.r, S.uj, mx, mb);
    }
    mx = block_reduce<true, float>(mx);
    if (kRhs<MODE>) mb = block_reduce<true, float>(mb);
    if (t == 0) {
      S.part[ONE_MAX * G + b0] = (double)mx;
      if (kRhs<MODE>) S.part[ONE_REF * G + b0] = (double)mb;
    }
    if (!grid_sync(S.bar, S.spins, target)) return false;
    m0 = grid_max(S.part + ONE_MAX * G);
    m1 = 0.0;
    if (kRhs<MODE>) {
      __syncthreads();  // grid_max's shared words
      m1 = grid_max(S.part + ONE_REF * G);
    }
    if (t == 0) {
      if (kRhs<MODE>) sc->ref = m1;
      outer_check(sc, m0, kRhs<MODE> ? fmax(S.R.tol, S.R.tol_rel * m1) : S.R.tol, S.R.maxit, 0, 0, 0);
    }
    __syncthreads();
    if (sc->outer_done) return true;
    while (!sc->inner_done) {
      if (!one_vcycle(S, target) || !grid_sync(S.bar, S.spins, target)) return false;
      T ru = 0, wu = 0;
      for (int b = b0; b < S.blocks; b += G) {
        Column c;
        if (block_column(S.R.cols, S.cbl, S.gx, b, t, c))
          cg_b_column(S.R.cols, c, S.R.code, S.u, S.r, S.w, ru, wu);
      }
      block_reduce2(ru, wu);
      if (t == 0) {
        S.part[ONE_RU * G + b0] = (double)ru;
        S.part[ONE_WU * G + b0] = (double)wu;
      }
      if (!grid_sync(S.bar, S.spins, target)) return false;
      grid_sums(S.part + ONE_RU * G, S.part + ONE_WU * G, m0, m1);
      if (t == 0) cg_scalars(sc, m0, m1, 0, 0);
      __syncthreads();
      if (sc->inner_done) break;  // a breakdown: no update
      const T alpha = (T)sc->alpha, beta = (T)sc->beta;
      const bool first = sc->round_iters == 0;
      T v;
      if (S.vec)
        v = cg_a_nodes<T, 16 / sizeof(T)>(S.N, k0, dk, S.R.code, S.x, S.r, S.u, S.uj, S.w, S.p, S.s, alpha, beta, first);
      else
        v = cg_a_nodes<T, 1>(S.N, k0, dk, S.R.code, S.x, S.r, S.u, S.uj, S.w, S.p, S.s, alpha, beta, first);
      v = block_reduce<true, T>(v);
      if (t == 0) S.part[ONE_MAX * G + b0] = (double)v;
      if (!grid_sync(S.bar, S.spins, target)) return false;
      m0 = grid_max(S.part + ONE_MAX * G);
      if (t == 0) cg_test(sc, m0, S.eta, S.tol_inner, S.R.maxit, 0, 0);
      __syncthreads();
    }
    if (sc->round_iters) {
      if (MODE == R_FX || MODE == R_FXG) correct_fx_nodes(S.N, k0, dk, (const float *)S.x, S.phifx, S.phi32, S.flag);
      else correct_nodes<T>(S.N, k0, dk, S.x, S.phi, S.phi32, S.phi_lo);
    }
    if (!grid_sync(S.bar, S.spins, target)) return false;
  }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 3 : 1) k_solve_one(const __grid_constant__ OneArgs<T> S) {
  __shared__ PoissonCtl sc;
  PoissonCtl *ctl = S.R.c;
  if (threadIdx.x == 0) {  // block 0 writes it back behind a barrier
    sc = *ctl;
    solve_reset(&sc);
  }
  __syncthreads();
  unsigned target = 0;
  const bool ok = one_solve<T, MODE>(S, &sc, target);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (ok && blockIdx.x == 0) {
      sc.one_iters += sc.solve_iters;
      sc.one_rounds += sc.rounds;
      sc.one_solves += 1;
      *ctl = sc;
    }
    // the block that leaves last (none waits any more) reports a wait that ran
    // out, after block 0 may have written the control block, and clears the
    // barrier (the ticket itself tells: a read of `dead` here is 1 us per solve)
    __threadfence();
    const unsigned ticket = atomicAdd(&S.bar->exits, ok ? 1u : 1u + kDeadExit);
    if (ticket % kDeadExit == gridDim.x - 1) {
      if (!ok || ticket >= kDeadExit) {
        __threadfence();
        ctl->sticky_status = LBE_ERR_CUDA;
      }
      S.bar->count = 0;
      S.bar->exits = 0;
      S.bar->dead = 0;
    }
  }
}

// ---------------------------------------------------------------------------
// kernel argument storage for graph nodes (values are copied at node creation)
struct Args {
  ResArgs R;  // the residual kernel's arguments, shared values among them
  int nblk, nblk_a;
  long long N;
  double eta, tol_inner;
  double *phi;               // FP64 iterate (FP64 form, linear solves)
  float *phi32, *phi_lo = nullptr;
  int64_t *phifx = nullptr;  // the FP32 form's fixed-point potential
  int *flag = nullptr;       // the FP32 form's range flags
  void *r, *u, *uj, *w, *x, *p, *s;
  double *part;
  dim3 flat;                 // grid of the pointwise kernels
};

cudaError_t add_kernel(cudaGraph_t gr, cudaGraphNode_t *last, void *func, dim3 grid, dim3 block, void **args) {
  cudaKernelNodeParams kp;
  memset(&kp, 0, sizeof(kp));
  kp.func = func;
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.kernelParams = args;
  cudaGraphNode_t n;
  cudaError_t e = cudaGraphAddKernelNode(&n, gr, *last ? last : nullptr, *last ? 1 : 0, &kp);
  if (e == cudaSuccess) *last = n;
  return e;
}

cudaError_t add_while(cudaGraph_t gr, cudaGraphNode_t *last, cudaGraphConditionalHandle h, cudaGraph_t *body) {
  // cudaGraphNodeParams has no default constructor: zeroed raw storage
  alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)];
  memset(raw, 0, sizeof(raw));
  cudaGraphNodeParams *np = reinterpret_cast<cudaGraphNodeParams *>(raw);
  np->type = cudaGraphNodeTypeConditional;
  np->conditional.handle = h;
  np->conditional.type = cudaGraphCondTypeWhile;
  np->conditional.size = 1;
  cudaGraphNode_t n;
  cudaError_t e = cudaGraphAddNode(&n, gr, *last ? last : nullptr, nullptr, *last ? 1 : 0, np);
  if (e == cudaSuccess) {
    *last = n;
    *body = np->conditional.phGraph_out[0];
  }
  return e;
}

template <typename T>
void fill_args(lbe_handle *h, Args &A) {
  PoissonWork &w = h->pw;
  const long long N = h->geo.N;
  T *base = (T *)w.vec;
  const ColLaunch L = make_cols(h->geo, h->phys.selfmask);
  ResArgs &R = A.R;
  R = ResArgs{};
  R.cols = L.c;
  R.g = h->geo;
  R.P = h->phys;
  R.P3 = h->p32;
  R.code = h->code;
  R.mask = h->mask;
  R.n64 = h->n;
  R.nq = h->q;
  R.phi = h->phi;
  R.phi_hi = h->phi32;
  R.phifx = h->phifx;
  R.nblk = (int)L.nblk();
  R.maxit = h->prm.poisson_max_iter;
  R.use_cond = 1;
  R.c = w.ctl;
  R.tol = h->prm.poisson_tol;
  {
    const double c6 = 6.0 * h->phys.four_pi_lb * h->p32.sd[0];  // 6 * 4 pi l_B * s, as two floats (R_FX)
    R.c6_hi = (float)c6;
    R.c6_lo = (float)(c6 - (double)R.c6_hi);
  }
  A.N = N;
  A.nblk = (int)L.nblk();
  A.flat = dim3((unsigned)std::min<long long>((N + kBlock - 1) / kBlock, kSolveBlocks));
  A.eta = sizeof(T) == 4 ? 1e-4 : 1e-9;
  // an inner solve need not go below a fraction of the outer tolerance:
  // 0.8 measured 2.15 CG iterations per step on the 64x64x256
  // electro-osmosis lattice against 2.9 at 0.25 and 2.4 at 0.5, with no
  // extra refinement round (the outer test still decides convergence)
  A.tol_inner = 0.8 * R.tol;
  A.phi = h->phi;
  A.phi32 = h->phi32;
  A.phifx = h->phifx;
  A.flag = h->flag;
  A.r = base;
  A.u = base + N;
  A.w = base + 2 * N;
  A.x = base + 3 * N;
  A.p = base + 4 * N;
  A.s = base + 5 * N;
  // the Jacobi vector r/diag: the V-cycle's input, or the preconditioned
  // vector itself without a hierarchy
  A.uj = h->mg.nlev >= 2 ? h->mg.t0 : A.u;
  A.part = w.partial;
}

template <typename T>
using ResKernel = void (*)(const ResArgs, T *, T *);
template <typename T>
ResKernel<T> res_kernel(const lbe_handle *h, const Args &A) {
  if (A.R.rhs) return A.R.phi_lo ? k_res<T, R_RHS_FF> : k_res<T, R_RHS>;
  if (h->prm.precision != LBE_FP32) return k_res<T, R_N64>;
  return h->p32.salt11 ? k_res<T, R_FX> : k_res<T, R_FXG>;
}
// The update handles 16 bytes of every vector at a time where the component
// stride (N values) keeps them aligned, else one value.
template <typename T>
using UpdateKernel = void (*)(long long, const uint8_t *, T *, T *, const T *, T *, const T *, T *, T *, int,
                              PoissonCtl *, double, double, int, cudaGraphConditionalHandle, int);
template <typename T>
UpdateKernel<T> update_kernel(long long N, int *vec) {
  constexpr int V = 16 / sizeof(T);
  *vec = N % V == 0 ? V : 1;
  return N % V == 0 ? k_cg_a<T, V> : k_cg_a<T, 1>;
}

template <typename T>
cudaError_t build_graph(lbe_handle *h, Args &A, cudaGraphExec_t *exec) {
  const ColLaunch L = make_cols(h->geo, h->phys.selfmask);
  const dim3 one(1), blk(kBlock);
  ResArgs &R = A.R;
  // the FP32 form's own solve corrects its fixed-point potential; the FP64
  // form and the linear solves correct an FP64 iterate
  const bool corr_fx = h->prm.precision == LBE_FP32 && !R.rhs;
  int vec = 1;
  const UpdateKernel<T> f_a = update_kernel<T>(A.N, &vec);
  const dim3 ga((unsigned)std::min<long long>((A.N / vec + kBlock - 1) / kBlock, kSolveBlocks));
  A.nblk_a = (int)ga.x;
  cudaGraph_t G = nullptr;
  cudaError_t e = cudaGraphCreate(&G, 0);
  if (e != cudaSuccess) return e;
  cudaGraphNode_t last = nullptr, lo = nullptr, li = nullptr;
  cudaGraph_t body_out = nullptr, body_in = nullptr;
  void *a_reset[] = {&R.c};
  void *a_res[] = {&R, &A.r, &A.uj};
  void *a_b[] = {&R.cols, &R.code, &A.u, &A.r, &A.w, &A.part, &A.nblk, &R.c, &R.hin, &R.use_cond};
  void *a_a[] = {&A.N, &R.code,   &A.x, &A.r,   &A.u,         &A.uj,    &A.w,   &A.p,
                 &A.s, &A.nblk_a, &R.c, &A.eta, &A.tol_inner, &R.maxit, &R.hin, &R.use_cond};
  void *a_cor[] = {&A.N, &A.x, &A.phi, &A.phi32, &A.phi_lo, &R.c};
  void *a_corfx[] = {&A.N, &A.x, &A.phifx, &A.phi32, &A.flag, &R.c};
  // reset -> while (not converged) { residual test -> while (CG) { V-cycle ->
  // stencil and dot products -> update and test } -> correct }.  The residual
  // test sets both conditions; in the pass where it converges the CG loop is
  // not entered and the correction returns at once.
  e = cudaGraphConditionalHandleCreate(&R.hout, G, 1, cudaGraphCondAssignDefault);
  if (e == cudaSuccess) e = add_kernel(G, &last, (void *)k_solve_reset, one, one, a_reset);
  if (e == cudaSuccess) e = add_while(G, &last, R.hout, &body_out);
  if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&R.hin, body_out, 0, 0);
  if (e == cudaSuccess) e = add_kernel(body_out, &lo, (void *)res_kernel<T>(h, A), L.grid, L.block, a_res);
  if (e == cudaSuccess) e = add_while(body_out, &lo, R.hin, &body_in);
  if (e == cudaSuccess && h->mg.nlev >= 2) e = mg_vcycle(h, A.r, A.uj, A.u, nullptr, body_in, &li, nullptr);
  if (e == cudaSuccess) e = add_kernel(body_in, &li, (void *)k_cg_b<T>, L.grid, L.block, a_b);
  if (e == cudaSuccess) e = add_kernel(body_in, &li, (void *)f_a, ga, blk, a_a);
  if (e == cudaSuccess)
    e = corr_fx ? add_kernel(body_out, &lo, (void *)k_correct_fx, A.flat, blk, a_corfx)
                : add_kernel(body_out, &lo, (void *)k_correct<T>, A.flat, blk, a_cor);
  if (e == cudaSuccess) e = cudaGraphInstantiate(exec, G, 0);
  cudaGraphDestroy(G);
  return e;
}

// host-driven fallback: the same kernels, polling the control block
template <typename T>
int solve_polled(lbe_handle *h, Args &A) {
  PoissonWork &w = h->pw;
  const ColLaunch L = make_cols(h->geo, h->phys.selfmask);
  cudaStream_t st = h->stream;
  ResArgs &R = A.R;
  R.use_cond = 0;
  int vec = 1;
  const UpdateKernel<T> f_a = update_kernel<T>(A.N, &vec);
  const dim3 ga((unsigned)std::min<long long>((A.N / vec + kBlock - 1) / kBlock, kSolveBlocks));
  const ResKernel<T> f_res = res_kernel<T>(h, A);
  const bool mg = h->mg.nlev >= 2;
  k_solve_reset<<<1, 1, 0, st>>>(R.c);
  h->launches += 1;
  auto poll = [&]() {
    cudaError_t e = cudaMemcpyAsync(w.ctl_host, w.ctl, sizeof(PoissonCtl), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) h->err = std::string("poisson: ") + cudaGetErrorString(e);
    return e;
  };
  for (int round = 0; round <= kMaxOuter + 1; ++round) {
    f_res<<<L.grid, L.block, 0, st>>>(R, (T *)A.r, (T *)A.uj);
    h->launches += 1;
    if (poll() != cudaSuccess) return LBE_ERR_CUDA;
    if (w.ctl_host->outer_done) break;
    const long long max_chunks = (long long)R.maxit / kChunk + 2;
    for (long long ch = 0; ch <= max_chunks && !w.ctl_host->inner_done; ++ch) {
      for (int k = 0; k < kChunk; ++k) {
        if (mg && mg_vcycle(h, A.r, A.uj, A.u, R.c, nullptr, nullptr, st) != cudaSuccess) return LBE_ERR_CUDA;
        k_cg_b<T><<<L.grid, L.block, 0, st>>>(R.cols, R.code, (T *)A.u, (T *)A.r, (T *)A.w, A.part, A.nblk, R.c, 0, 0);
        f_a<<<ga, kBlock, 0, st>>>(A.N, R.code, (T *)A.x, (T *)A.r, (T *)A.u, (T *)A.uj, (T *)A.w, (T *)A.p, (T *)A.s,
                                   (int)ga.x, R.c, A.eta, A.tol_inner, R.maxit, 0, 0);
      }
      h->launches += 2 * kChunk;
      if (poll() != cudaSuccess) return LBE_ERR_CUDA;
    }
    if (h->prm.precision == LBE_FP32 && !R.rhs)
      k_correct_fx<<<A.flat, kBlock, 0, st>>>(A.N, (const float *)A.x, A.phifx, A.phi32, A.flag, R.c);
    else
      k_correct<T><<<A.flat, kBlock, 0, st>>>(A.N, (const T *)A.x, A.phi, A.phi32, A.phi_lo, R.c);
    h->launches += 1;
  }
  return cudaGetLastError() == cudaSuccess ? LBE_OK : LBE_ERR_CUDA;
}

// The solve as one cooperative launch; false where the lattice, its hierarchy
// or the device does not take it (the graph or the polled loop does).
template <typename T>
bool solve_one(lbe_handle *h, const Args &A, int *rc) {
  PoissonWork &w = h->pw;
  if (!w.one_ok || A.N > kOneNodes) return false;
  OneArgs<T> S;
  if (!mg_one_args(h, &S.V)) return false;
  const void *f;
  if (sizeof(T) == 8)
    f = (const void *)k_solve_one<double, R_N64>;
  else if (A.R.rhs) {
    if (!A.phi_lo) return false;
    f = (const void *)k_solve_one<float, R_RHS_FF>;
  } else
    f = h->p32.salt11 ? (const void *)k_solve_one<float, R_FX> : (const void *)k_solve_one<float, R_FXG>;
  const ColLaunch L = make_cols(h->geo, h->phys.selfmask);
  S.R = A.R;
  S.R.use_cond = 0;
  S.r = (T *)A.r;
  S.u = (T *)A.u;
  S.uj = (T *)A.uj;
  S.w = (T *)A.w;
  S.x = (T *)A.x;
  S.p = (T *)A.p;
  S.s = (T *)A.s;
  S.phi = A.phi;
  S.phi32 = A.phi32;
  S.phi_lo = A.phi_lo;
  S.phifx = A.phifx;
  S.flag = A.flag;
  S.part = w.one_part;
  S.bar = (GridBar *)w.one_bar;
  S.spins = w.one_spins;
  S.N = A.N;
  S.eta = A.eta;
  S.tol_inner = A.tol_inner;
  S.cbl = 0;
  while ((1u << S.cbl) < L.block.x) ++S.cbl;
  S.gx = (int)L.grid.x;
  S.blocks = (int)L.nblk();
  S.vec = A.N % (16 / sizeof(T)) == 0;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kBlock, 0);
  if (e == cudaSuccess && per_sm > 0) {
    per_sm = std::min(per_sm, kOnePerSM<T>);
    const int G = std::min(std::min(std::max(S.blocks, std::min((S.V.ndense + 7) / 8, sms)), per_sm * sms), kOneBlocks);
    void *args[] = {&S};
    e = cudaLaunchCooperativeKernel(f, dim3((unsigned)G), dim3(kBlock), args, 0, h->stream);
    if (e == cudaSuccess) {
      h->launches += 1;
      *rc = LBE_OK;
      return true;
    }
  }
  cudaGetLastError();  // not on this device: the other paths
  w.one_ok = false;
  return false;
}

template <typename T>
int solve_t(lbe_handle *h) {
  PoissonWork &w = h->pw;
  {
    Args A;
    int rc;
    fill_args<T>(h, A);
    if (solve_one<T>(h, A, &rc)) return rc;
  }
  // one graph per solute buffer (flow-off steps swap the two buffers)
  const void *key = h->prm.precision == LBE_FP32 ? (const void *)h->q : (const void *)h->n;
  int slot = -1;
  for (int k = 0; k < 2; ++k)
    if (w.exec[k] && w.exec_key[k] == key) slot = k;
  if (slot < 0 && w.graph_ok) {
    slot = !w.exec[0] ? 0 : (!w.exec[1] ? 1 : 0);
    if (w.exec[slot]) cudaGraphExecDestroy(w.exec[slot]);
    w.exec[slot] = nullptr;
    Args A;
    fill_args<T>(h, A);
    cudaError_t e = build_graph<T>(h, A, &w.exec[slot]);
    if (e != cudaSuccess) {
      cudaGetLastError();  // clear the error; use the polled loop from now on
      w.graph_ok = false;
      w.exec[slot] = nullptr;
      slot = -1;
    } else {
      w.exec_key[slot] = key;
    }
  }
  if (slot >= 0) {
    cudaError_t e = cudaGraphLaunch(w.exec[slot], h->stream);
    if (e != cudaSuccess) {
      h->err = std::string("poisson graph launch: ") + cudaGetErrorString(e);
      return LBE_ERR_CUDA;
    }
    return LBE_OK;
  }
  Args A;
  fill_args<T>(h, A);
  return solve_polled<T>(h, A);
}

}  // namespace

cudaError_t poisson_alloc(lbe_handle *h) {
  PoissonWork &w = h->pw;
  const long long N = h->geo.N;
  w.L = make_launch(h->geo, kSolveBlocks);
  const size_t tsz = h->prm.precision == LBE_FP32 ? sizeof(float) : sizeof(double);
  cudaError_t e;
  if ((e = cudaMalloc(&w.vec, tsz * 6 * N)) != cudaSuccess) return e;
  const size_t nblk = (size_t)make_cols(h->geo, h->phys.selfmask).nblk();
  if ((e = cudaMalloc(&w.partial, sizeof(double) * 2 * nblk)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.phi_prev, sizeof(double) * kHist * N)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&w.ctl, sizeof(PoissonCtl))) != cudaSuccess) return e;
  if ((e = cudaMemset(w.ctl, 0, sizeof(PoissonCtl))) != cudaSuccess) return e;
  if ((e = cudaMallocHost(&w.ctl_host, sizeof(PoissonCtl))) != cudaSuccess) return e;
  // LBE_POISSON_GRAPH=0 runs the solves from the host loop (same kernels),
  // e.g. for profilers that do not follow conditional graph nodes
  const char *env = getenv("LBE_POISSON_GRAPH");
  w.graph_ok = !(env && env[0] == '0');
  int dev = 0, coop = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
  w.one_ok = coop && w.graph_ok && N <= kOneNodes;
  const char *spins = getenv("LBE_SOLVE_SPINS");
  w.one_spins = spins ? std::max(0, atoi(spins)) : kSpinLimit;
  if (w.one_ok) {
    if ((e = cudaMalloc(&w.one_part, sizeof(double) * 3 * kOneBlocks)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&w.one_bar, sizeof(GridBar))) != cudaSuccess) return e;
    if ((e = cudaMemset(w.one_bar, 0, sizeof(GridBar))) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void poisson_free(lbe_handle *h) {
  PoissonWork &w = h->pw;
  for (int k = 0; k < 2; ++k)
    if (w.exec[k]) cudaGraphExecDestroy(w.exec[k]);
  if (w.exec_lin) cudaGraphExecDestroy(w.exec_lin);
  cudaFree(w.vec);
  cudaFree(w.partial);
  cudaFree(w.phi_prev);
  cudaFree(w.one_part);
  cudaFree(w.one_bar);
  cudaFree(w.ctl);
  if (w.ctl_host) cudaFreeHost(w.ctl_host);
  w = PoissonWork{};
}

void poisson_drop_graphs(lbe_handle *h) {
  PoissonWork &w = h->pw;
  for (int k = 0; k < 2; ++k) {
    if (w.exec[k]) cudaGraphExecDestroy(w.exec[k]);
    w.exec[k] = nullptr;
    w.exec_key[k] = nullptr;
  }
  if (w.exec_lin) cudaGraphExecDestroy(w.exec_lin);
  w.exec_lin = nullptr;
  w.lin_key[0] = w.lin_key[1] = w.lin_key[2] = nullptr;
}

int poisson_solve_linear(lbe_handle *h, const double *rhs, double *x, double tol_abs, double tol_rel, float *x_hi,
                         float *x_lo) {
  if (h->prm.precision != LBE_FP32) {
    h->err = "linear solve: FP32 form only";
    return LBE_ERR_STATE;
  }
  PoissonWork &w = h->pw;
  Args A;
  fill_args<float>(h, A);
  A.R.rhs = rhs;
  A.R.phi = A.phi = x;
  A.R.phi_hi = A.phi32 = x_hi;
  A.R.phi_lo = A.phi_lo = x_hi ? x_lo : nullptr;
  if (A.phi_lo) {  // the split of the starting x; the corrections keep it current
    k_correct<float><<<A.flat, kBlock, 0, h->stream>>>(A.N, nullptr, x, x_hi, x_lo, nullptr);
    if (cudaGetLastError() != cudaSuccess) return LBE_ERR_CUDA;
  }
  A.R.tol = tol_abs;
  A.R.tol_rel = tol_rel;
  A.tol_inner = 0.25 * tol_abs;
  int rc;
  if (solve_one<float>(h, A, &rc)) return rc;
  if (!w.graph_ok) return solve_polled<float>(h, A);
  if (!w.exec_lin || w.lin_key[0] != rhs || w.lin_key[1] != x || w.lin_key[2] != x_hi) {
    if (w.exec_lin) cudaGraphExecDestroy(w.exec_lin);
    w.exec_lin = nullptr;
    cudaError_t e = build_graph<float>(h, A, &w.exec_lin);
    if (e != cudaSuccess) {
      h->err = std::string("linear solve graph: ") + cudaGetErrorString(e);
      w.exec_lin = nullptr;
      return LBE_ERR_CUDA;
    }
    w.lin_key[0] = rhs;
    w.lin_key[1] = x;
    w.lin_key[2] = x_hi;
  }
  cudaError_t e = cudaGraphLaunch(w.exec_lin, h->stream);
  if (e != cudaSuccess) {
    h->err = std::string("linear solve graph launch: ") + cudaGetErrorString(e);
    return LBE_ERR_CUDA;
  }
  return LBE_OK;
}

int poisson_enqueue(lbe_handle *h, bool extrapolate, bool extrapolated) {
  PoissonWork &w = h->pw;
  if (lone_fluid_node(h->geo, h->no_solid)) {
    h->err = "poisson: non-finite residual";
    return LBE_ERR_NONFINITE;
  }
  if (extrapolate) {
    if (!extrapolated) {
      if (h->prm.precision == LBE_FP32)
        k_extrapolate_fx<<<w.L.grid, w.L.block, 0, h->stream>>>(h->geo, w.L.zpt, h->mask, h->phifx,
                                                                (int64_t *)w.phi_prev, h->phi32, w.history);
      else
        k_extrapolate<<<w.L.grid, w.L.block, 0, h->stream>>>(h->geo, w.L.zpt, h->mask, h->phi, w.phi_prev, nullptr,
                                                           nullptr, w.history);
      h->launches += 1;
    }
    if (w.history < kHist) w.history += 1;
  } else {
    w.history = 0;
  }
  if (h->prm.precision == LBE_FP32) {
    h->phi64_stale = true;  // the solve moves the fixed-point potential
    return solve_t<float>(h);
  }
  return solve_t<double>(h);
}

int poisson_status(lbe_handle *h, lbe_stats *st, long long *kernels) {
  PoissonWork &w = h->pw;
  cudaError_t e = cudaMemcpyAsync(w.ctl_host, w.ctl, sizeof(PoissonCtl), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    h->err = std::string("poisson: ") + cudaGetErrorString(e);
    return LBE_ERR_CUDA;
  }
  const PoissonCtl &c = *w.ctl_host;
  if (st) {
    st->poisson_iters = c.total_iters;
    st->poisson_solves = (int)c.solves;
    st->poisson_max_iters = (int)(c.solve_iters > c.max_solve_iters ? c.solve_iters : c.max_solve_iters);
    st->poisson_residual = c.res;
  }
  if (kernels && w.graph_ok) {  // the polled and the single-kernel solves are counted as they are launched
    // kernels of the graph path: per solve the reset; per residual test the
    // test and the correction; per iteration V-cycle (with multigrid),
    // stencil and update
    const long long vc = mg_kernels_per_cycle(h);
    *kernels = (c.solves - c.one_solves) + 2 * (c.total_rounds - c.one_rounds) +
               (2 + vc) * (c.total_iters - c.one_iters);
  }
  if (c.sticky_status == LBE_ERR_CUDA) {
    h->err = "poisson: a wait between the solve's blocks ran out";
    return LBE_ERR_CUDA;
  }
  if (c.sticky_status == LBE_ERR_NOCONVERGE || c.status == LBE_ERR_NOCONVERGE) {
    h->err = "poisson: no convergence within poisson_max_iter";
    return LBE_ERR_NOCONVERGE;
  }
  if (c.sticky_status == LBE_ERR_NONFINITE || c.status == LBE_ERR_NONFINITE) {
    h->err = "poisson: non-finite residual";
    return LBE_ERR_NONFINITE;
  }
  return LBE_OK;
}

cudaError_t poisson_reset_stats(lbe_handle *h) { return cudaMemsetAsync(h->pw.ctl, 0, sizeof(PoissonCtl), h->stream); }


}  // namespace lbe
