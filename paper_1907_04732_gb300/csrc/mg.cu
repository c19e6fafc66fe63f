// Geometric multigrid preconditioner of the Poisson correction solve, in the
// form's own precision: FP32 vectors and operators in the FP32 form, FP64
// throughout in the FP64 form (whose solve took 40-190 Jacobi iterations per
// step before it had the hierarchy, 3-7 with it: 64x64x256 electro-osmosis
// 12.6 -> 0.97 ms, 128x128x4 coax 1.55 -> 0.44, 4x4x64 plates 0.78 -> 0.14).
//
// The CG of the Poisson solve (poisson.cu) needs u = M r with M ~ A^-1; the
// plain Jacobi choice M = D^-1 leaves it O(L) iterations on an L-long gap.
// Here M is one symmetric V-cycle; the hierarchy, smoother and correction
// are described with their per-node arithmetic in mg_device.cuh.  Any
// symmetric positive definite M leaves the CG fixed point unchanged.
//
// Kernels per V-cycle: the pre-smoothing sweep from zero (e = omega r/diag)
// is evaluated on the fly where it is needed (restriction, prolongation), so
// a cycle over levels 0..L is L restrictions, the coarsest solve and L fused
// prolongation+post-smoothing kernels.  The
// coarsest level is solved exactly (its inverse, formed once on the host; a
// lattice without solid nodes takes the pseudo-inverse): a weak coarse solve costs CG
// iterations (on the 64x64x256 electro-osmosis lattice 3.2 per step with 32
// Jacobi sweeps, 2.6 with 64 or 128 sweeps or the exact solve).
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "vcycle.cuh"

namespace lbe {

namespace {

using namespace mgd;

__device__ __forceinline__ bool lnode(const MgLevel &L, int &x, int &y, int &z, int &r) {
  x = blockIdx.x * blockDim.x + threadIdx.x;
  y = blockIdx.y * blockDim.y + threadIdx.y;
  z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= L.nx || y >= L.ny || z >= L.nz) return false;
  r = x + L.nx * (y + L.ny * z);
  return true;
}

// --- set-up: level-0 inverse diagonal, Galerkin coarse operators -------------
// level 1 from the fine lattice (mask-defined operator)
template <typename T>
__global__ void k_galerkin0(const Geo g, uint32_t selfmask, const uint32_t *__restrict__ mask, const MgLevel C,
                            T *__restrict__ A) {
  int X, Y, Z, I;
  if (!lnode(C, X, Y, Z, I)) return;
  T a[27];
  galerkin0_row(g, selfmask, mask, C, X, Y, Z, a);
#pragma unroll
  for (int d = 0; d < 27; ++d) A[d * C.S + I] = a[d];
}

// level l+1 from level l (27-point)
template <typename T>
__global__ void k_galerkin(const MgLevel F, const T *__restrict__ AF, const MgLevel C, T *__restrict__ A) {
  int X, Y, Z, I;
  if (!lnode(C, X, Y, Z, I)) return;
  T a[27];
  galerkin_row(F, AF, C, X, Y, Z, a);
#pragma unroll
  for (int d = 0; d < 27; ++d) A[d * C.S + I] = a[d];
}

// --- V-cycle kernels (bodies in vcycle.cuh) ------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_restrict0(const Cols F, const uint8_t *__restrict__ code,
                                                   const T *__restrict__ r, const T *__restrict__ u, const MgLevel C,
                                                   const T *__restrict__ WC, T *__restrict__ rc, T *__restrict__ zc,
                                                   const RestrictMap M, const PoissonCtl *c) {
  if (c && c->inner_done) return;
  restrict0_block(F, code, r, u, C, WC, rc, zc, M, (int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z);
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict(const MgLevel F, const T *__restrict__ AF,
                                                  const T *__restrict__ r, const T *__restrict__ zf,
                                                  const MgLevel C, const T *__restrict__ WC,
                                                  T *__restrict__ rc, T *__restrict__ zc, int txl, int Z0,
                                                  const PoissonCtl *c) {
  if (c && c->inner_done) return;
  restrict_block(F, AF, r, zf, C, WC, rc, zc, txl, (int)blockIdx.x, (int)blockIdx.y, Z0 + (int)blockIdx.z);
}

// fused prolongation + post-smoothing on a 27-point level
template <typename T>
__global__ void k_post(const MgLevel L, const T *__restrict__ A, const T *__restrict__ W, const T *__restrict__ r,
                       const T *__restrict__ z, const MgLevel C, const T *__restrict__ ec,
                       T *__restrict__ out, const PoissonCtl *c) {
  if (c && c->inner_done) return;
  int X, Y, Z, I;
  if (!lnode(L, X, Y, Z, I)) return;
  // W null: omega/diag by division.  FP64: the division costs more than its
  // stored value (float measured 2 % of the solve the other way round: one
  // more load, so it reads W only where the weight is not kOmega)
  out[I] = W ? post_value_w(L, A, W[I], r, z, C, ec, X, Y, Z) : post_value_z(L, A, r, z, C, ec, X, Y, Z);
}

template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 3) k_post0(const Cols F, const uint8_t *__restrict__ code,
                                               const uint32_t *__restrict__ mask, const T *__restrict__ r,
                                               const T *__restrict__ u, const MgLevel C, const T *__restrict__ ec,
                                               T *__restrict__ out, const PoissonCtl *c) {
  if (c && c->inner_done) return;
  Column col;
  if (column_of(F, col)) post0_column(F, col, code, mask, r, u, C, ec, out);
}

// coarsest level solved exactly: e = A^-1 r with the inverse formed at
// set-up, one warp per row (a fixed summation order)
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_direct(int N, const T *__restrict__ Ainv, const T *__restrict__ r,
                                                       T *__restrict__ e, const PoissonCtl *c) {
  if (c && c->inner_done) return;
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row < N) inverse_row(row, N, Ainv, r, e);
}

// coarsest level in one block
template <typename T>
__global__ void __launch_bounds__(kCoarseMax) k_coarsest(const MgLevel L, const T *__restrict__ A,
                                                         const T *__restrict__ r, T *__restrict__ e,
                                                         const PoissonCtl *c) {
  if (c && c->inner_done) return;
  __shared__ T buf[2][kCoarseMax];
  coarsest_solve(L, A, r, e, buf);
}

// --- the bottom of the V-cycle as one matrix ------------------------------------
// On the levels from ld down the V-cycle is a fixed linear map e = M r of at
// most kDenseMax nodes.  Its matrix is formed at set-up, one block per column
// running those levels on a unit vector in shared memory, and applied by
// one kernel, one warp per row.  As kernels of their own a restriction, the
// coarsest solve and a post-smoothing take 11 us of launch, ramp and drain
// for a few thousand nodes of work; one 16-block cluster with barriers
// between the phases took as long (14 us, and 4 us more per iteration in the
// graph); the product with a 2048 x 2048 matrix (17 MB, held by L2) takes 6 us,
// with a 1024 x 1024 one 3.6 us.
template <typename T>
constexpr int kDenseMax = sizeof(T) == 4 ? 3072 : 1024;  // FP64: its pipe does 304 products a cycle
constexpr int kDenseThreads = 512;

template <typename T>
struct BottomLevel {
  MgLevel L;
  const T *A, *W;
};
template <typename T>
struct BottomArgs {
  BottomLevel<T> lv[kMaxLevels];
  int ld, nl, stride;
  const T *cinv;
  T *M;
};

template <typename T>
__global__ void __launch_bounds__(kDenseThreads) k_dense_form(const BottomArgs<T> G) {
  extern __shared__ unsigned char sh_raw[];
  T *sh = reinterpret_cast<T *>(sh_raw);  // per level: r, then e, z computed on the fly (z = W r)
  const int col = blockIdx.x;
  T *r = sh;
  for (int i = threadIdx.x; i < G.lv[G.ld].L.N; i += blockDim.x) r[i] = i == col ? (T)1 : (T)0;
  __syncthreads();
  for (int l = G.ld; l + 1 < G.nl; ++l) {
    const MgLevel F = G.lv[l].L, C = G.lv[l + 1].L;
    const T *A = G.lv[l].A, *W = G.lv[l].W;
    T *rc = r + F.N;
    for (int I = threadIdx.x; I < C.N; I += blockDim.x) {
      int X, Y, Z;
      level_coords(C, I, X, Y, Z);
      T v = 0;
      for (int ch = 0; ch < 8; ++ch) {
        int x, y, z;
        if (!child_of(C, X, Y, Z, ch, F.nx, F.ny, F.nz, x, y, z)) continue;
        const int i = x + F.nx * (y + F.ny * z);
        T s = 0;
        for (int q = 0; q < 27; ++q) {
          const int j = wrap(x + q % 3 - 1, F.nx) +
                        F.nx * (wrap(y + (q / 3) % 3 - 1, F.ny) + F.ny * wrap(z + q / 9 - 1, F.nz));
          s = fma(A[q * F.S + i], W[j] * r[j], s);
        }
        v += r[i] - s;
      }
      rc[I] = v;
    }
    r = rc;
    __syncthreads();
  }
  const int Nc = G.lv[G.nl - 1].L.N;
  T *e = r + Nc;
  for (int i = threadIdx.x; i < Nc; i += blockDim.x) {
    T s = 0;
    for (int j = 0; j < Nc; ++j) s = fma(G.cinv[(size_t)j * Nc + i], r[j], s);  // symmetric: coalesced over i
    e[i] = s;
  }
  __syncthreads();
  for (int l = G.nl - 2; l >= G.ld; --l) {
    const MgLevel F = G.lv[l].L, C = G.lv[l + 1].L;
    const T *A = G.lv[l].A, *W = G.lv[l].W;
    r -= F.N;
    T *ef = e + C.N;
    for (int i = threadIdx.x; i < F.N; i += blockDim.x) {
      int x, y, z;
      level_coords(F, i, x, y, z);
      T s = 0;
      for (int q = 0; q < 27; ++q) {
        const int jx = wrap(x + q % 3 - 1, F.nx), jy = wrap(y + (q / 3) % 3 - 1, F.ny), jz = wrap(z + q / 9 - 1, F.nz);
        const int j = jx + F.nx * (jy + F.ny * jz);
        s = fma(A[q * F.S + i], fma((T)kAlpha, e[agg_index(C, jx, jy, jz)], W[j] * r[j]), s);
      }
      const T w = W[i];
      ef[i] = w != (T)0 ? fma((T)kAlpha, e[agg_index(C, x, y, z)], w * r[i]) + w * (r[i] - s) : (T)0;
    }
    e = ef;
    __syncthreads();
  }
  // column col; M is symmetric, stored as rows for the product
  const int N = G.lv[G.ld].L.N;
  for (int i = threadIdx.x; i < G.stride; i += blockDim.x)
    G.M[(size_t)col * G.stride + i] = i < N ? e[i] : (T)0;
}

// e = M r
template <typename T>
__global__ void __launch_bounds__(256) k_dense(int N, int stride, const T *__restrict__ M, const T *__restrict__ r,
                                               T *__restrict__ e, const PoissonCtl *c) {
  if (c && c->inner_done) return;
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row < N) dense_row(row, stride, M, r, e);
}

// omega/diag of a level (0 for a node without fluid)
template <typename T>
__global__ void k_weights(int N, float omega, const T *__restrict__ A13, T *__restrict__ W) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const T d = A13[i];
  W[i] = d != (T)0 ? (T)omega / d : (T)0;
}

dim3 lgrid(const MgLevel &L, dim3 &block) {
  const Geo g{L.nx, L.ny, L.nz, 0, 0, 0, L.N};
  const Launch la = make_launch(g);
  block = la.block;
  return la.grid;
}

// launches of the restriction into level L
constexpr int kGridZ = 65535;
int restrict_launches(const MGLevel &L) { return (L.nz + kGridZ - 1) / kGridZ; }

MgLevel level_dev(const MGLevel &L) { return MgLevel{L.nx, L.ny, L.nz, L.sx, L.sy, L.sz, (int)L.N, L.N}; }


}  // namespace

// Inverse of the coarsest level's operator from its 27-point rows (host,
// FP64): the operator restricted to the nodes with a non-zero diagonal
// (aggregates holding fluid) is assembled densely, factored A = L L^T
// (Cholesky) and inverted; rows and columns of the other nodes are zero,
// as the Jacobi sweeps leave them.  False when the operator is not
// symmetric positive definite to working accuracy: the sweeps are used then.
//
// singular: a lattice without solid nodes, whose operator annihilates
// constants.  The rounding of the FP32 form's rows decides whether its last
// pivot is positive, and an inverse that passed would answer a constant with
// 1e7 times what it answers anything else (of 20 such lattices, half failed to
// converge in some of their solves).  The pseudo-inverse is formed instead,
//   A+ = (A + (c/n) 1 1^T)^-1 - 1/(c n) 1 1^T   for any c > 0.
template <typename T>
static bool coarse_inverse_t(const mgd::MgLevel &L, const std::vector<T> &A27, std::vector<T> &inv, bool singular) {
  const int N = L.N;
  std::vector<int> act;  // active node -> level index
  std::vector<int> pos(N, -1);
  for (int i = 0; i < N; ++i)
    if (A27[13 * (size_t)N + i] != (T)0) {
      pos[i] = (int)act.size();
      act.push_back(i);
    }
  const int n = (int)act.size();
  inv.assign((size_t)N * N, (T)0);
  if (n == 0 || (singular && n == 1)) return true;
  std::vector<double> M((size_t)n * n, 0.0);
  for (int a = 0; a < n; ++a) {
    const int I = act[a];
    const int X = I % L.nx, Y = (I / L.nx) % L.ny, Z = I / (L.nx * L.ny);
    for (int q = 0; q < 27; ++q) {
      const T v = A27[(size_t)q * N + I];
      if (v == (T)0) continue;
      auto wr = [](int c, int m) { return c < 0 ? c + m : (c >= m ? c - m : c); };
      const int J = wr(X + q % 3 - 1, L.nx) + L.nx * (wr(Y + (q / 3) % 3 - 1, L.ny) + L.ny * wr(Z + q / 9 - 1, L.nz));
      if (pos[J] < 0) continue;  // a zero of the correction
      M[(size_t)a * n + pos[J]] += (double)v;
    }
  }
  double dmax = 0.0, asym = 0.0, amax = 0.0;
  for (int a = 0; a < n; ++a) {
    dmax = std::max(dmax, M[(size_t)a * n + a]);
    for (int b = 0; b < n; ++b) {
      amax = std::max(amax, std::fabs(M[(size_t)a * n + b]));
      asym = std::max(asym, std::fabs(M[(size_t)a * n + b] - M[(size_t)b * n + a]));
    }
  }
  if (!(dmax > 0.0) || asym > 1e-5 * amax) return false;
  if (singular)
    for (double &m : M) m += dmax / n;
  // Cholesky A = U^T U by rows of U, then the inverse's lower triangle X from
  // U^T Y = I and U X = Y.  Every inner loop runs along contiguous rows, with
  // independent elements: the compiler vectorises it, and none waits for the
  // sum before it (dot products down the columns of a 256-node level took 9 ms,
  // as long as forty steps of the lattice that needs it).
  for (int j = 0; j < n; ++j) {
    double *u = &M[(size_t)j * n];
    for (int k = 0; k < j; ++k) {
      const double *uk = &M[(size_t)k * n];
      const double f = uk[j];
      for (int i = j; i < n; ++i) u[i] -= f * uk[i];
    }
    if (!(u[j] > 1e-10 * dmax)) return false;
    const double ujj = std::sqrt(u[j]), s = 1.0 / ujj;
    u[j] = ujj;
    for (int i = j + 1; i < n; ++i) u[i] *= s;
  }
  std::vector<double> X((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i) {
    double *x = &X[(size_t)i * n];
    x[i] = 1.0;
    for (int k = 0; k < i; ++k) {
      const double f = M[(size_t)k * n + i], *xk = &X[(size_t)k * n];
      for (int c = 0; c <= k; ++c) x[c] -= f * xk[c];
    }
    const double s = 1.0 / M[(size_t)i * n + i];
    for (int c = 0; c <= i; ++c) x[c] *= s;
  }
  for (int i = n - 1; i >= 0; --i) {
    double *x = &X[(size_t)i * n];
    for (int k = i + 1; k < n; ++k) {
      const double f = M[(size_t)i * n + k], *xk = &X[(size_t)k * n];
      for (int c = 0; c <= i; ++c) x[c] -= f * xk[c];
    }
    const double s = 1.0 / M[(size_t)i * n + i];
    for (int c = 0; c <= i; ++c) {
      x[c] *= s;
      const double v = singular ? x[c] - 1.0 / (dmax * n) : x[c];
      inv[(size_t)act[i] * N + act[c]] = inv[(size_t)act[c] * N + act[i]] = (T)v;
    }
  }
  return true;
}
bool mgd::coarse_inverse(const MgLevel &L, const std::vector<float> &A27, std::vector<float> &inv, bool singular) {
  return coarse_inverse_t(L, A27, inv, singular);
}

// the matrix of the V-cycle from the first level of at most kDenseMax nodes
// down (levels above the coarsest, whose inverse is already a matrix)
template <typename T>
static cudaError_t form_dense(lbe_handle *h) {
  MGWork &mg = h->mg;
  int ld = mg.nlev - 1;
  while (ld > 1 && mg.lv[ld - 1].N <= kDenseMax<T>) --ld;
  if (ld == mg.nlev - 1) return cudaSuccess;
  const int N = (int)mg.lv[ld].N;
  constexpr int V = 16 / sizeof(T);
  BottomArgs<T> G;
  G.ld = ld;
  G.nl = mg.nlev;
  G.stride = (N + V - 1) / V * V;
  G.cinv = (const T *)mg.cinv;
  size_t shared = 0;  // at most 47.6 KB (a chain: 3072 + 1536 + ... + 192 nodes)
  for (int l = ld; l < mg.nlev; ++l) {
    G.lv[l] = BottomLevel<T>{level_dev(mg.lv[l]), (const T *)mg.lv[l].A, (const T *)mg.lv[l].W};
    shared += 2 * sizeof(T) * (size_t)mg.lv[l].N;
  }
  cudaError_t e = cudaMalloc(&mg.dense, sizeof(T) * (size_t)N * G.stride);
  if (e != cudaSuccess) return e;
  G.M = (T *)mg.dense;
  k_dense_form<T><<<(unsigned)N, kDenseThreads, shared, h->stream>>>(G);
  mg.ld = ld;
  mg.stride = G.stride;
  return cudaGetLastError();
}

// build the hierarchy for the current geometry (after the link mask)
template <typename T>
static cudaError_t mg_setup_t(lbe_handle *h) {
  MGWork &mg = h->mg;
  mg_free(h);
  const Geo &g = h->geo;
  MgLevel shp[kMaxLevels];
  mg.nlev = level_shapes(g.nx, g.ny, g.nz, shp);
  if (mg.nlev == 0) return cudaSuccess;  // plain Jacobi preconditioning
  for (int l = 1; l < mg.nlev; ++l) {
    MGLevel &L = mg.lv[l];
    L.nx = shp[l].nx;
    L.ny = shp[l].ny;
    L.nz = shp[l].nz;
    L.sx = shp[l].sx;
    L.sy = shp[l].sy;
    L.sz = shp[l].sz;
    L.N = shp[l].N;
  }
  cudaError_t e = cudaMalloc(&mg.t0, sizeof(T) * g.N);
  for (int l = 1; l < mg.nlev && e == cudaSuccess; ++l) {
    MGLevel &L = mg.lv[l];
    e = cudaMalloc(&L.A, sizeof(T) * 27 * L.N);
    if (e == cudaSuccess) e = cudaMalloc(&L.W, sizeof(T) * L.N);
    // k_dense reads r in 16-byte words: padded, the padding zero
    if (e == cudaSuccess) e = cudaMalloc(&L.r, sizeof(T) * (L.N + 4));
    if (e == cudaSuccess) e = cudaMemsetAsync((T *)L.r + L.N, 0, sizeof(T) * 4, h->stream);
    if (e == cudaSuccess) e = cudaMalloc(&L.e, sizeof(T) * L.N);
    if (e == cudaSuccess) e = cudaMalloc(&L.z, sizeof(T) * L.N);
  }
  if (e != cudaSuccess) {
    mg_free(h);
    return e;
  }
  for (int l = 1; l < mg.nlev; ++l) {
    const MgLevel C = level_dev(mg.lv[l]);
    dim3 blk;
    const dim3 grd = lgrid(C, blk);
    if (l == 1)
      k_galerkin0<T><<<grd, blk, 0, h->stream>>>(g, h->phys.selfmask, h->mask, C, (T *)mg.lv[1].A);
    else
      k_galerkin<T><<<grd, blk, 0, h->stream>>>(level_dev(mg.lv[l - 1]), (const T *)mg.lv[l - 1].A, C,
                                                (T *)mg.lv[l].A);
  }
  cudaError_t le = cudaGetLastError();
  if (le != cudaSuccess) return le;
  for (int l = 1; l < mg.nlev; ++l)
    k_weights<T><<<(unsigned)((mg.lv[l].N + 255) / 256), 256, 0, h->stream>>>(
        (int)mg.lv[l].N, jacobi_weight(g, kOmega), (const T *)mg.lv[l].A + 13 * mg.lv[l].N, (T *)mg.lv[l].W);
  le = cudaGetLastError();
  if (le != cudaSuccess) return le;
  mg.ld = mg.nlev - 1;
  // the coarsest level is solved exactly where its operator is SPD
  // (LBE_MG_DIRECT=0: Jacobi sweeps everywhere)
  const char *denv = getenv("LBE_MG_DIRECT");
  if (!(denv && denv[0] == '0')) {
    const MGLevel &Lc = mg.lv[mg.nlev - 1];
    std::vector<T> a27((size_t)27 * Lc.N), inv;
    le = cudaMemcpyAsync(a27.data(), Lc.A, sizeof(T) * a27.size(), cudaMemcpyDeviceToHost, h->stream);
    if (le == cudaSuccess) le = cudaStreamSynchronize(h->stream);
    if (le != cudaSuccess) return le;
    if (coarse_inverse_t(level_dev(Lc), a27, inv, h->no_solid)) {
      le = cudaMalloc(&mg.cinv, sizeof(T) * inv.size());
      if (le == cudaSuccess)
        le = cudaMemcpyAsync(mg.cinv, inv.data(), sizeof(T) * inv.size(), cudaMemcpyHostToDevice, h->stream);
      if (le == cudaSuccess) le = cudaStreamSynchronize(h->stream);  // inv is released on return
      if (le != cudaSuccess) return le;
      return form_dense<T>(h);
    }
  }
  return cudaSuccess;
}
cudaError_t mg_setup(lbe_handle *h) {
  return h->prm.precision == LBE_FP32 ? mg_setup_t<float>(h) : mg_setup_t<double>(h);
}

void mg_free(lbe_handle *h) {
  MGWork &mg = h->mg;
  for (int l = 0; l < kMaxLevels; ++l) {
    cudaFree(mg.lv[l].A);
    cudaFree(mg.lv[l].W);
    cudaFree(mg.lv[l].r);
    cudaFree(mg.lv[l].e);
    cudaFree(mg.lv[l].z);
  }
  cudaFree(mg.t0);
  cudaFree(mg.cinv);
  cudaFree(mg.dense);
  mg = MGWork{};
}

// u = M r as a sequence of kernels, either launched on the stream or added to
// a graph (gr != nullptr) after *last
template <typename T>
static cudaError_t mg_vcycle_t(lbe_handle *h, const void *r0, const void *uj, void *u0, const PoissonCtl *c,
                               cudaGraph_t gr, cudaGraphNode_t *last, cudaStream_t st) {
  MGWork &mg = h->mg;
  const int nl = mg.nlev;
  // finest-level kernels: the solve's launch
  ColLaunch L0 = make_cols(h->geo, h->phys.selfmask);
  // kernel arguments live in these arrays until the nodes are created or the
  // kernels launched
  struct Node {
    void *f;
    dim3 grid, block;
    void *args[12];
  };
  std::vector<Node> nodes;
  std::vector<MgLevel> lv(kMaxLevels);
  std::vector<const void *> ptr;
  ptr.reserve(512);  // no reallocation: the kernel arguments point into it
  auto P = [&](const void *v) -> void * {
    ptr.push_back(v);
    return &ptr.back();
  };
  for (int l = 1; l < nl; ++l) lv[l] = level_dev(mg.lv[l]);
  // down: restrictions (pre-smoothing on the fly)
  RestrictMap M;
  const dim3 rg0 = make_restrict_map(h->geo, lv[1], M);
  nodes.push_back(Node{(void *)k_restrict0<T>, rg0, dim3(256),
                       {&L0.c, P(h->code), P(r0), P(uj), &lv[1], P(mg.lv[1].W), P(mg.lv[1].r), P(mg.lv[1].z), &M,
                        P(c)}});
  // the level whose V-cycle is one matrix (or the coarsest)
  const int lk = mg.ld;
  int txl[kMaxLevels];
  std::vector<int> z0;
  size_t restricts = 0;
  for (int l = 1; l < lk; ++l) restricts += restrict_launches(mg.lv[l + 1]);
  z0.reserve(restricts);  // no reallocation: the kernel arguments point into it
  for (int l = 1; l < lk; ++l) {
    const MGLevel &Lc = mg.lv[l + 1];
    const dim3 rg = restrict_tiles(lv[l + 1], txl[l]);
    // a launch per kGridZ planes, the limit of a grid's z axis (a loop over the
    // planes in the kernel took 7 % longer per solve of 256x256x128 nodes)
    for (int k = 0; k < restrict_launches(Lc); ++k) {
      z0.push_back(k * kGridZ);
      nodes.push_back(Node{(void *)k_restrict<T>, dim3(rg.x, rg.y, std::min<unsigned>(rg.z - z0.back(), kGridZ)),
                           dim3(256),
                           {&lv[l], P(mg.lv[l].A), P(mg.lv[l].r), P(mg.lv[l].z), &lv[l + 1], P(Lc.W), P(Lc.r),
                            P(Lc.z), &txl[l], &z0.back(), P(c)}});
    }
  }
  // coarsest: exact (inverse) or Jacobi sweeps
  int ncoarse = (int)mg.lv[nl - 1].N;
  int ndense = (int)mg.lv[lk].N;
  if (mg.dense) {
    nodes.push_back(Node{(void *)k_dense<T>, dim3((unsigned)((ndense + 7) / 8)), dim3(256),
                         {&ndense, &mg.stride, P(mg.dense), P(mg.lv[lk].r), P(mg.lv[lk].e), P(c)}});
  } else if (mg.cinv)
    nodes.push_back(Node{(void *)k_coarse_direct<T>, dim3((unsigned)((ncoarse + 7) / 8)), dim3(256),
                         {&ncoarse, P(mg.cinv), P(mg.lv[nl - 1].r), P(mg.lv[nl - 1].e), P(c)}});
  else
    nodes.push_back(Node{(void *)k_coarsest<T>, dim3(1), dim3(kCoarseMax),
                         {&lv[nl - 1], P(mg.lv[nl - 1].A), P(mg.lv[nl - 1].r), P(mg.lv[nl - 1].e), P(c)}});
  // up: fused prolongation + post-smoothing
  const bool use_w = sizeof(T) == 8 || jacobi_weight(h->geo, kOmega) != kOmega;
  for (int l = lk - 1; l >= 1; --l) {
    dim3 blk;
    const dim3 grd = lgrid(lv[l], blk);
    nodes.push_back(Node{(void *)k_post<T>, grd, blk,
                         {&lv[l], P(mg.lv[l].A), P(use_w ? mg.lv[l].W : nullptr), P(mg.lv[l].r), P(mg.lv[l].z), &lv[l + 1],
                          P(mg.lv[l + 1].e), P(mg.lv[l].e), P(c)}});
  }
  nodes.push_back(Node{(void *)k_post0<T>, L0.grid, L0.block,
                       {&L0.c, P(h->code), P(h->mask), P(r0), P(uj), &lv[1], P(mg.lv[1].e), P(u0), P(c)}});
  cudaError_t e = cudaSuccess;
  for (Node &n : nodes) {
    if (gr) {
      cudaKernelNodeParams kp;
      memset(&kp, 0, sizeof(kp));
      kp.func = n.f;
      kp.gridDim = n.grid;
      kp.blockDim = n.block;
      kp.kernelParams = n.args;
      cudaGraphNode_t nd;
      e = cudaGraphAddKernelNode(&nd, gr, *last ? last : nullptr, *last ? 1 : 0, &kp);
      if (e != cudaSuccess) return e;
      *last = nd;
    } else {
      e = cudaLaunchKernel(n.f, n.grid, n.block, n.args, 0, st);
      if (e != cudaSuccess) return e;
      h->launches += 1;
    }
  }
  return e;
}
cudaError_t mg_vcycle(lbe_handle *h, const void *r0, const void *uj, void *u0, const PoissonCtl *c, cudaGraph_t gr,
                      cudaGraphNode_t *last, cudaStream_t st) {
  return h->prm.precision == LBE_FP32 ? mg_vcycle_t<float>(h, r0, uj, u0, c, gr, last, st)
                                      : mg_vcycle_t<double>(h, r0, uj, u0, c, gr, last, st);
}

template <typename T>
static bool one_args(lbe_handle *h, VCycleArgs<T> *V) {
  const MGWork &mg = h->mg;
  if (mg.nlev < 2 || !(mg.dense || mg.cinv)) return false;
  *V = VCycleArgs<T>{};
  V->ld = mg.ld;
  V->ndense = (int)mg.lv[mg.ld].N;
  V->stride = mg.dense ? mg.stride : 0;
  V->mat = (const T *)(mg.dense ? mg.dense : mg.cinv);
  for (int l = 1; l <= mg.ld; ++l) {
    const MGLevel &L = mg.lv[l];
    V->lv[l] = level_dev(L);
    V->A[l] = (const T *)L.A;
    V->W[l] = (const T *)L.W;
    V->r[l] = (T *)L.r;
    V->z[l] = (T *)L.z;
    V->e[l] = (T *)L.e;
    if (l > 1) {
      const dim3 t = restrict_tiles(V->lv[l], V->txl[l - 1]);
      V->rx[l - 1] = (int)t.x;
      V->ry[l - 1] = (int)t.y;
      V->rz[l - 1] = (int)t.z;
    }
  }
  const dim3 g = make_restrict_map(h->geo, V->lv[1], V->M);
  V->g0x = (int)g.x;
  V->g0y = (int)g.y;
  V->g0z = (int)g.z;
  return true;
}
bool mg_one_args(lbe_handle *h, VCycleArgs<float> *V) { return one_args(h, V); }
bool mg_one_args(lbe_handle *h, VCycleArgs<double> *V) { return one_args(h, V); }

// kernels of one V-cycle (launch accounting of the graph path)
int mg_kernels_per_cycle(const lbe_handle *h) {
  const MGWork &mg = h->mg;
  if (mg.nlev < 2) return 0;
  int n = 2 * mg.ld + 1;
  for (int l = 2; l <= mg.ld; ++l) n += restrict_launches(mg.lv[l]) - 1;
  return n;
}

}  // namespace lbe
