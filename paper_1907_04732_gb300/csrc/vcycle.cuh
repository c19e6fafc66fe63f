// Block and thread bodies of the V-cycle's kernels, shared by the kernels of
// mg.cu (one launch each) and the single-kernel solve of poisson.cu (all of
// them as phases).  Pointers to values that a phase of the same launch writes
// carry no __restrict__: those must not become read-only-cache loads.
#pragma once

#include "march.cuh"
#include "mg_device.cuh"

namespace lbe {
namespace mgd {

// Level 1: a fluid child's pre-smoothed residual is r - omega A u, u = r/diag
// being the Jacobi vector the CG formed.  A thread marches (march.cuh) a fine
// column over the planes of Kc coarse ones; a warp covers 2^xl x 2^yl columns
// (aligned pairs along every halved axis) of 2^zl chunks, so that the
// children of a coarse node meet in the thread (z) and in two shuffles (x, y),
// a fixed order.
struct RestrictMap {
  int xl, yl, zl;  // lanes 2^xl x 2^yl x 2^zl
  int wy;          // warps of a block along y (the rest along z)
  int Kc;          // coarse planes per thread
};
// where thread t of block (bx, by, bz) works: its fine column and first coarse
// plane, and its place in the warp along x and y
struct RestrictLane {
  int lx, ly, x, y, Z0;
};
__host__ __device__ __forceinline__ RestrictLane restrict_lane(const RestrictMap &M, int t, int bx, int by, int bz) {
  const int lane = t & 31, w = t >> 5;
  RestrictLane l;
  l.lx = lane & ((1 << M.xl) - 1);
  l.ly = (lane >> M.xl) & ((1 << M.yl) - 1);
  l.x = (bx << M.xl) + l.lx;
  l.y = ((by * M.wy + w % M.wy) << M.yl) + l.ly;
  l.Z0 = (((bz * (8 / M.wy) + w / M.wy) << M.zl) + (lane >> (M.xl + M.yl))) * M.Kc;
  return l;
}
template <typename T>
__device__ __forceinline__ void restrict0_block(const Cols &F, const uint8_t *code, const T *r, const T *u,
                                                const MgLevel &C, const T *WC, T *rc, T *zc, const RestrictMap &M,
                                                int bx, int by, int bz) {
  const RestrictLane l = restrict_lane(M, (int)threadIdx.x, bx, by, bz);
  const int lx = l.lx, ly = l.ly, x = l.x, y = l.y, Z0 = l.Z0;
  const bool own = x < F.nx && y < F.ny && Z0 < C.nz;
  const int p = x + F.nx * y;
  const PlaneOffs o = plane_offs(F.nx, F.ny, x, y);
  ZMarch<T> m;
  int z = Z0 << C.sz;
  const int zend = min((Z0 + M.Kc) << C.sz, F.nz);
  if (own) m.begin(u, o, p, F.plane, F.nz, z);
#pragma unroll 1
  for (int k = 0; k < M.Kc; ++k) {  // every lane runs the same iterations (the shuffles)
    const int Z = Z0 + k;
    const bool write = own && Z < C.nz && !(C.sx & lx & 1) && !(C.sy & ly & 1);
    const int I = (x >> C.sx) + C.nx * ((y >> C.sy) + C.ny * Z);
    const T wd = write ? WC[I] : (T)0;
    T v = 0;
    if (own && Z < C.nz) {
      for (int h = 0; h <= C.sz && z < F.nz; ++h, ++z) {
        if (F.ahead && z + 1 + F.ahead < zend) {
          prefetch_l2(u + m.j + F.plane * (1 + F.ahead));
          prefetch_l2(r + m.j + F.plane * F.ahead);
          prefetch_l2(code + m.j + F.plane * F.ahead);
        }
        T u0;
        int i;
        const T nsum = m.step(u, o, p, F.plane, F.nz, z, u0, i);
        const int cd = code[i];
        const T res = r[i] - (T)F.omega * ((T)((cd & kCodeDiag) + F.selfw) * u0 - nsum) * (T)(1.0 / 6.0);
        v += cd ? res : (T)0;
      }
    }
    if (C.sx) v += __shfl_xor_sync(0xffffffffu, v, 1);
    if (C.sy) v += __shfl_xor_sync(0xffffffffu, v, 1 << M.xl);
    if (write) {
      rc[I] = v;
      zc[I] = wd * v;
    }
  }
}

// lanes along x, a pair of rows, the rest along z; returns the grid of
// 256-thread blocks
inline dim3 make_restrict_map(const Geo &g, const MgLevel &L1, RestrictMap &M, int Kc = 0) {
  M.yl = L1.sy;
  M.xl = 0;
  while ((1 << M.xl) < g.nx && M.xl < 5 - M.yl) ++M.xl;
  M.zl = 5 - M.xl - M.yl;
  const int xt = (g.nx + (1 << M.xl) - 1) >> M.xl, yt = (g.ny + (1 << M.yl) - 1) >> M.yl;
  M.wy = yt < 8 ? pow2_at_least(yt) : 8;
  const int zc = (8 / M.wy) << M.zl, yb = (yt + M.wy - 1) / M.wy;  // chunks per block, blocks along y
  M.Kc = Kc ? Kc : planes_per_thread((long long)xt * yb, L1.nz, zc, 1 + L1.sz);
  const int per = zc * M.Kc;
  return dim3((unsigned)xt, (unsigned)yb, (unsigned)((L1.nz + per - 1) / per));
}

// tiles of k_restrict: 32 coarse nodes per block, 2^txl along X (at most 32)
// and the rest along Y, one plane per block
inline dim3 restrict_tiles(const MgLevel &C, int &txl) {
  txl = 0;
  while ((1 << txl) < C.nx && txl < 5) ++txl;
  return dim3((unsigned)((C.nx + (1 << txl) - 1) >> txl), (unsigned)((C.ny + (32 >> txl) - 1) / (32 >> txl)),
              (unsigned)C.nz);
}

// Restriction between coarse levels with 8 threads per coarse node (one per
// child) and a fixed-order shuffle sum of the children's pre-smoothed
// residuals.  A block covers a tile of 32
// coarse nodes (2^txl along X, the rest along Y; lanes 8k..8k+7 the children
// of one coarse node, child index = lane % 8 as in child_of) of one plane:
// coordinates come from the block and lane indices, with no division.
template <typename T>
__device__ __forceinline__ void restrict_block(const MgLevel &F, const T *AF, const T *r, const T *zf, const MgLevel &C,
                                               const T *WC, T *rc, T *zc, int txl, int bx, int by, int bz) {
  const int ch = threadIdx.x & 7, j = threadIdx.x >> 3;
  const int X = (bx << txl) + (j & ((1 << txl) - 1));
  const int Y = by * (32 >> txl) + (j >> txl), Z = bz;
  const bool own = X < C.nx && Y < C.ny;
  const int I = X + C.nx * (Y + C.ny * Z);
  const T wd = ch == 0 && own ? WC[I] : (T)0;
  int x, y, z;
  T v = 0;
  if (own && child_of(C, X, Y, Z, ch, F.nx, F.ny, F.nz, x, y, z)) v = presmoothed_res_z(F, AF, r, zf, x, y, z);
  v = sum8(v);
  if (ch == 0 && own) {
    rc[I] = v;
    zc[I] = wd * v;
  }
}

// fused prolongation + post-smoothing on the finest level:
// t = omega u + alpha P e_1 (fluid nodes), out = t + omega (r - A t)/diag.
// The neighbour sum of u is marched; that of P e_1 likewise, with the coarse
// array's offsets (a column's neighbours lie in its own aggregate or the next
// one) and each coarse plane's sums kept while the fine planes stay in it.
// Next to a wall, P e_1 is nonzero on the solid neighbours too and the links
// are taken one by one.
template <typename T>
__device__ __forceinline__ void post0_column(const Cols &F, const Column &col, const uint8_t *code, const uint32_t *mask,
                                             const T *r, const T *u, const MgLevel &C, const T *ec, T *out) {
  const int X = col.x >> C.sx, Y = col.y >> C.sy, cplane = C.nx * C.ny;
  PlaneOffs q;  // coarse offsets of the in-plane neighbours' aggregates
  q.xm = ((col.x + col.o.xm) >> C.sx) - X;
  q.xp = ((col.x + col.o.xp) >> C.sx) - X;
  q.ym = C.nx * (((col.y == 0 ? F.ny - 1 : col.y - 1) >> C.sy) - Y);
  q.yp = C.nx * (((col.y == F.ny - 1 ? 0 : col.y + 1) >> C.sy) - Y);
  const int P = X + C.nx * Y;
  const T om = (T)F.omega, al = (T)kAlpha;
  ZMarch<T> m;
  m.begin(u, col.o, col.p, F.plane, F.nz, col.z0);
  int Z = col.z0 >> C.sz;
  T c0, s0, d0, c1, s1, d1, below;
  {
    T cb, sb, db;
    const int Zb = (col.z0 == 0 ? F.nz - 1 : col.z0 - 1) >> C.sz;
    plane_sums(ec, q, P + cplane * Zb, cb, sb, db);
    below = 2 * cb + sb;
  }
  plane_sums(ec, q, P + cplane * Z, c0, s0, d0);
  auto node = [&](int z) {
    if (F.ahead && z + 1 + F.ahead < col.z1) {
      prefetch_l2(u + m.j + F.plane * (1 + F.ahead));
      prefetch_l2(r + m.j + F.plane * F.ahead);
      prefetch_l2(code + m.j + F.plane * F.ahead);
      prefetch_l2(ec + P + cplane * ((z + 1 + F.ahead) >> C.sz));
    }
    T u0;
    int i;
    const int Zn = (z + 1 == F.nz ? 0 : z + 1) >> C.sz;
    if (Zn != Z) {
      plane_sums(ec, q, P + cplane * Zn, c1, s1, d1);
    } else {
      c1 = c0;
      s1 = s0;
      d1 = d0;
    }
    const T nu = m.step(u, col.o, col.p, F.plane, F.nz, z, u0, i);
    T ne = (2 * s0 + d0) + (below + (2 * c1 + s1));
    const int cd = code[i];
    T v = 0;
    if (cd) {
      if (cd & kCodeWall) {
        const uint32_t mk = mask[i];
        const int Zm = (z == 0 ? F.nz - 1 : z - 1) >> C.sz;
        ne = 0;
#pragma unroll
        for (int l = 1; l < kQ; ++l) {
          const int dx = cx_of(l), dy = cy_of(l), dz = cz_of(l);
          const int a = P + (dx < 0 ? q.xm : (dx > 0 ? q.xp : 0)) + (dy < 0 ? q.ym : (dy > 0 ? q.yp : 0)) +
                        cplane * (dz < 0 ? Zm : (dz > 0 ? Zn : Z));
          if (mk & (1u << (l - 1))) ne += (T)(c2_of(l) == 1 ? 2 : 1) * ec[a];
        }
      }
      const T d6 = (T)(cd & kCodeDiag);
      const T t = om * u0 + al * c0;
      const T s6 = om * nu + al * ne - (T)F.selfw * t;
      const T res6 = (T)6 * r[i] - (d6 * t - s6);
      v = t + om * (sizeof(T) == 4 ? (T)__fdividef((float)res6, (float)d6) : res6 * (T)(1.0 / 6.0) * inv_diag<T>(cd));
    }
    out[i] = v;
    below = 2 * c0 + s0;
    c0 = c1;
    s0 = s1;
    d0 = d1;
    Z = Zn;
  };
  if (F.ahead) {  // from HBM: several planes' loads in flight
#pragma unroll 2
    for (int z = col.z0; z < col.z1; ++z) node(z);
  } else {
#pragma unroll 1
    for (int z = col.z0; z < col.z1; ++z) node(z);
  }
}

// one row of e = A^-1 r by a warp, the inverse's rows unpadded
template <typename T>
__device__ __forceinline__ void inverse_row(int row, int N, const T *Ainv, const T *r, T *e) {
  const int lane = threadIdx.x & 31;
  const T *a = Ainv + (size_t)row * N;
  T s = 0;
  for (int j = lane; j < N; j += 32) s = fma(a[j], r[j], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) e[row] = s;
}

// one row of e = M r by a warp; rows of `stride` values (a multiple of 16
// bytes, zero-padded, as r is)
template <typename T>
__device__ __forceinline__ void dense_row(int row, int stride, const T *M, const T *r, T *e) {
  constexpr int V = 16 / sizeof(T);
  struct alignas(16) Vec {
    T v[V];
  };
  const int lane = threadIdx.x & 31;
  const Vec *a = reinterpret_cast<const Vec *>(M + (size_t)row * stride);
  const Vec *b = reinterpret_cast<const Vec *>(r);
  T s[V] = {};
#pragma unroll 8
  for (int k = lane; k < stride / V; k += 32) {
    const Vec av = a[k], bv = b[k];
#pragma unroll
    for (int q = 0; q < V; ++q) s[q] = fma(av.v[q], bv.v[q], s[q]);
  }
  T t = s[0];
#pragma unroll
  for (int q = 1; q < V; ++q) t += s[q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) e[row] = t;
}

// the V-cycle's levels and matrices as kernel arguments of the single-kernel
// solve (filled by mg_one_args in mg.cu)
template <typename T>
struct VCycleArgs {
  int ld;  // the level solved by one matrix
  int ndense, stride;  // its nodes; row stride of its matrix (0: the coarsest level's inverse)
  const T *mat;
  MgLevel lv[kMaxLevels];
  const T *A[kMaxLevels], *W[kMaxLevels];
  T *r[kMaxLevels], *z[kMaxLevels], *e[kMaxLevels];
  RestrictMap M;
  int g0x, g0y, g0z;                  // blocks of the restriction into level 1
  int txl[kMaxLevels];                // restrictions l -> l + 1 (restrict_tiles)
  int rx[kMaxLevels], ry[kMaxLevels], rz[kMaxLevels];
};

}  // namespace mgd

// false: no hierarchy, or a coarsest level solved by Jacobi sweeps
bool mg_one_args(lbe_handle *h, mgd::VCycleArgs<float> *V);
bool mg_one_args(lbe_handle *h, mgd::VCycleArgs<double> *V);

}  // namespace lbe
