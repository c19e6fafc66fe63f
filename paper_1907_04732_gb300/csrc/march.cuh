// Column-marching launch of the single lattice's finest-level stencil kernels.
//
// A thread owns one (x, y) column position of the lattice and walks a chunk
// of consecutive z planes.  The 19-point Laplacian's link weights are 2
// (axis) and 1 (diagonal) over 6, so with, per plane, c the value at the
// column, s the sum of its four in-plane axis neighbours and d that of its
// four in-plane diagonal ones, the weighted neighbour sum of plane z is
//   6 sum_l w_l v_l = 2 s(z) + d(z) + T(z-1) + T(z+1),   T = 2 c + s.
// T(z-1) is carried from plane to plane and plane z+1 becomes the next centre:
// nine loads and ten additions per node instead of eighteen neighbours, each
// with its own address and weight.  Every neighbour is read unconditionally:
// the solve's correction vectors hold zeros on solid nodes (Dirichlet), so no
// link needs its mask bit, and no load waits for another one.  Kernel times
// on the 64x64x256 lattice, before and after: CG stencil 21 -> 12.5 us,
// residual 24 -> 16, restriction 13 -> 9, prolongation and post-smoothing
// 12 -> 10.5 (one kernel).
//
// Column positions are flattened (p = x + nx y): a block covers 256
// consecutive positions, or all positions of a smaller plane for several z
// chunks, so that a ragged nx leaves no thread idle (a launch tiled over x
// rounds nx up to a power of two).
#pragma once

#include "mg_device.cuh"

namespace lbe {

// Division of unsigned 32-bit integers by a run-time invariant divisor d >= 1
// by a multiplication and shifts (Granlund and Montgomery, "Division by
// invariant integers using multiplication", PLDI 1994, Sec. 4): with
// l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1,
// q = (t + ((n - t) >> min(l,1))) >> max(l-1,0), t = high word of m n.
struct FastDiv {
  uint32_t d, m;
  int sh1, sh2;
};

inline FastDiv make_fastdiv(uint32_t d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  FastDiv f;
  f.d = d;
  f.m = (uint32_t)(((((uint64_t)1 << l) - d) << 32) / d + 1);
  f.sh1 = l < 1 ? l : 1;
  f.sh2 = l > 1 ? l - 1 : 0;
  return f;
}

__host__ __device__ __forceinline__ uint32_t fdiv(const FastDiv &f, uint32_t n) {
#ifdef __CUDA_ARCH__
  const uint32_t t = __umulhi(f.m, n);
#else
  const uint32_t t = (uint32_t)(((uint64_t)f.m * n) >> 32);
#endif
  return (t + ((n - t) >> f.sh1)) >> f.sh2;
}

// Node codes of the solve's kernels (one byte per node): 6 x the diagonal of
// -lap_mod at a fluid node (6..48; links of a node to itself left out), bit 7
// set when one of its 18 links joins a solid node; 0 on solid nodes.
constexpr int kCodeDiag = 0x7f, kCodeWall = 0x80;

// 1/diag from a node's code (6 diag; 0 on a solid node, as its inverse).  A
// double division takes a dozen instructions on the narrow FP64 pipe, so the
// FP64 form reads the inverses from a table.
struct InvDiag {
  double v[49];
  constexpr InvDiag() : v() {
    for (int k = 1; k < 49; ++k) v[k] = 1.0 / ((double)k * (1.0 / 6.0));
  }
};
static __constant__ InvDiag kInvDiag = InvDiag();
template <typename T>
__device__ __forceinline__ T inv_diag(int code) {
  const int d6 = code & kCodeDiag;
  if (sizeof(T) == 8) return (T)kInvDiag.v[d6];
  return (T)(d6 ? 1.f / ((float)d6 * (1.f / 6.f)) : 0.f);
}

// lattices above this size (about 30 bytes of solve vectors per node in use
// at a time) do not stay in the 129 MB L2
constexpr long long kPrefetchNodes = 3 << 20;

// A lattice cut into columns of K planes
struct Cols {
  int nx, ny, nz, plane;  // plane = nx ny
  int K;                  // planes per thread
  int selfw;              // 6 x the weights of the links that join a node to itself
  int ahead;              // planes to prefetch ahead of the march (0: none)
  float omega;            // the V-cycle's Jacobi weight (jacobi_weight)
  FastDiv fnx;
};
struct ColLaunch {
  Cols c{};
  dim3 grid, block;
  long long nblk() const { return (long long)grid.x * grid.y; }
};

// Planes per thread for nz planes of gx column blocks (zb chunks a block): the
// K that minimises waves x (K + 3), the march costing about three planes of
// latency besides its K (two planes to start, the reduction at the end), with
// kResident blocks at once (five per SM at 48 registers).  On the 256^3
// lattice, with the L2 prefetch (Cols::ahead), K = 32 takes the CG stencil
// from 113 to 86 us, the post-smoothing from 222 to 136 and the restriction
// from 125 to 94 against K = 64 in 1024 blocks; at 64x64x256 the two agree
// (12.4-13.7 us).
constexpr int kResident = 760;
inline int planes_per_thread(long long gx, int nz, int zb, int unit = 1) {
  long long best = 0;
  int bestK = 1;
  for (int K = 1; K <= 64; ++K) {
    const long long gy = (nz + (long long)K * zb - 1) / ((long long)K * zb);
    const long long cost = (gx * gy + kResident - 1) / kResident * (K * unit + 3);
    if (K == 1 || cost < best) {
      best = cost;
      bestK = K;
    }
    if (gy == 1) break;
  }
  return bestK;
}

// The V-cycle's Jacobi weight.  A lattice with one axis longer than one node
// is a chain: its Jacobi-scaled operator reaches 2, where the weight 1 that
// suits wider lattices (at most 1.6) does not damp the alternating mode at
// all, and 2/3 is the best for the upper half of its modes.
inline float jacobi_weight(const Geo &g, float omega) {
  return (g.nx > 1) + (g.ny > 1) + (g.nz > 1) == 1 ? omega * (2.f / 3.f) : omega;
}

// K: planes per thread (0: chosen for this lattice alone); nodes: of all the
// lattices that a kernel works on (0: this one alone)
inline ColLaunch make_cols(const Geo &g, uint32_t selfmask, int K = 0, long long nodes = 0) {
  ColLaunch L;
  L.c.nx = g.nx;
  L.c.ny = g.ny;
  L.c.nz = g.nz;
  L.c.plane = g.nx * g.ny;
  L.c.fnx = make_fastdiv((uint32_t)g.nx);
  L.c.selfw = 0;
  for (int i = 1; i < kQ; ++i)
    if (selfmask & (1u << (i - 1))) L.c.selfw += c2_of(i) == 1 ? 2 : 1;
  const int cb = L.c.plane < 256 ? pow2_at_least(L.c.plane) : 256, zb = 256 / cb;
  const long long gx = ((long long)L.c.plane + cb - 1) / cb;
  if (K == 0) K = planes_per_thread(gx, g.nz, zb);
  L.c.K = K;
  // a lattice whose vectors exceed L2 is read from HBM: its latency is
  // covered by prefetching the columns' next planes into L2
  L.c.ahead = (nodes ? nodes : g.N) > kPrefetchNodes ? 3 : 0;
  L.c.omega = jacobi_weight(g, mgd::kOmega);
  L.block = dim3((unsigned)cb, (unsigned)zb);
  L.grid = dim3((unsigned)gx, (unsigned)((g.nz + (long long)K * zb - 1) / ((long long)K * zb)));
  return L;
}

// in-plane neighbour offsets of a column, periodic wrap included
struct PlaneOffs {
  int xm, xp, ym, yp;
};
__host__ __device__ __forceinline__ PlaneOffs plane_offs(int nx, int ny, int x, int y) {
  PlaneOffs o;
  o.xm = x == 0 ? nx - 1 : -1;
  o.xp = x == nx - 1 ? 1 - nx : 1;
  o.ym = y == 0 ? (ny - 1) * nx : -nx;
  o.yp = y == ny - 1 ? (1 - ny) * nx : nx;
  return o;
}

// this thread's column and chunk [z0, z1); false when it has none
struct Column {
  int p, x, y, z0, z1;
  PlaneOffs o;
};
// (p: the column, chunk: which K planes of it)
__host__ __device__ __forceinline__ bool column_at(const Cols &C, int p, int chunk, Column &c) {
  c.p = p;
  c.z0 = chunk * C.K;
  if (c.p >= C.plane || c.z0 >= C.nz) return false;
  c.z1 = c.z0 + C.K < C.nz ? c.z0 + C.K : C.nz;
  c.y = (int)fdiv(C.fnx, (uint32_t)c.p);
  c.x = c.p - c.y * C.nx;
  c.o = plane_offs(C.nx, C.ny, c.x, c.y);
  return true;
}

// thread t of block b, the blocks numbered in one dimension: gx across the
// columns (2^cbl of them each), then up the chunks
__host__ __device__ __forceinline__ bool block_column(const Cols &C, int cbl, int gx, int b, int t, Column &c) {
  return column_at(C, ((b % gx) << cbl) + (t & ((1 << cbl) - 1)), (b / gx) * (256 >> cbl) + (t >> cbl), c);
}

__device__ __forceinline__ bool column_of(const Cols &C, Column &c) {
  return column_at(C, (int)(blockIdx.x * blockDim.x + threadIdx.x), (int)(blockIdx.y * blockDim.y + threadIdx.y), c);
}

// neighbour offsets of node (column, z) for the per-link forms
__device__ __forceinline__ Offs col_offs(const PlaneOffs &o, int plane, int nz, int z) {
  Offs f;
  f.xm = o.xm;
  f.xp = o.xp;
  f.ym = o.ym;
  f.yp = o.yp;
  f.zm = z == 0 ? (nz - 1) * plane : -plane;
  f.zp = z == nz - 1 ? (1 - nz) * plane : plane;
  return f;
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <typename V>
__device__ __forceinline__ void plane_sums(const V *v, const PlaneOffs &o, int j, V &c, V &s, V &d) {
  const V *q = v + j;
  c = q[0];
  s = (q[o.xm] + q[o.xp]) + (q[o.ym] + q[o.yp]);
  d = (q[o.xm + o.ym] + q[o.xp + o.ym]) + (q[o.xm + o.yp] + q[o.xp + o.yp]);
}

// one column's march over the planes of v
template <typename V>
struct ZMarch {
  V c, s, d, below;  // of the current plane; T of the plane below it
  int j;             // its node
  __device__ __forceinline__ void begin(const V *v, const PlaneOffs &o, int p, int plane, int nz, int z) {
    V c0, s0, d0;
    j = p + plane * z;
    plane_sums(v, o, z == 0 ? p + plane * (nz - 1) : j - plane, c0, s0, d0);
    below = 2 * c0 + s0;
    plane_sums(v, o, j, c, s, d);
  }
  // 6 sum_l w_l v_l of plane z, then plane z + 1 becomes the current one
  // (straight-line code: the loads of several unrolled steps go out together)
  __device__ __forceinline__ V step(const V *v, const PlaneOffs &o, int p, int plane, int nz, int z, V &centre,
                                    int &at) {
    const int k = z + 1 == nz ? p : j + plane;
    V c1, s1, d1;
    plane_sums(v, o, k, c1, s1, d1);
    const V sum = (2 * s + d) + (below + (2 * c1 + s1));
    centre = c;
    at = j;
    below = 2 * c + s;
    c = c1;
    s = s1;
    d = d1;
    j = k;
    return sum;
  }
};

}  // namespace lbe
