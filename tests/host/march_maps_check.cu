// Host check of the index functions that the column-marching kernels call
// themselves (block_column, column_at, plane_offs in march.cuh; restrict_lane in
// vcycle.cuh): no GPU is used.  For ragged shapes, with the planes per thread
// that the single lattice chooses and with those that a batch hands over (1 to
// 16, half of it for the restriction), every node lies in one chunk, offsets
// name the periodic neighbours, every coarse node is written by one thread that
// meets its other columns in the two shuffles.  The Python test parses the lines.
#include <cstdio>
#include <vector>

#include "../../paper_1907_04732_gb300/csrc/vcycle.cuh"

using namespace lbe;

static bool columns(const Geo &g, int K) {
  const ColLaunch L = make_cols(g, 0u, K, K ? 1 << 24 : 0);
  int cbl = 0;
  while ((1u << cbl) < L.block.x) ++cbl;
  if ((1u << cbl) * L.block.y != 256u) return false;
  std::vector<int> seen((size_t)g.N, 0);
  for (int b = 0; b < (int)L.nblk(); ++b)
    for (int t = 0; t < 256; ++t) {
      Column c, d;
      // the two-dimensional launch of the same block (column_of)
      const int bx = b % (int)L.grid.x, by = b / (int)L.grid.x;
      const int tx = t % (int)L.block.x, ty = t / (int)L.block.x;
      const bool in = block_column(L.c, cbl, (int)L.grid.x, b, t, c);
      if (in != column_at(L.c, bx * (int)L.block.x + tx, by * (int)L.block.y + ty, d)) return false;
      if (!in) continue;
      if (c.p != d.p || c.z0 != d.z0 || c.z1 != d.z1 || c.z1 <= c.z0 || c.z1 > g.nz) return false;
      if (c.x < 0 || c.x >= g.nx || c.p != c.x + g.nx * c.y) return false;
      if (c.p + c.o.xm != nbr(g, c.x, c.y, 0, -1, 0, 0) || c.p + c.o.xp != nbr(g, c.x, c.y, 0, 1, 0, 0) ||
          c.p + c.o.ym != nbr(g, c.x, c.y, 0, 0, -1, 0) || c.p + c.o.yp != nbr(g, c.x, c.y, 0, 0, 1, 0) ||
          c.p + c.o.xp + c.o.ym != nbr(g, c.x, c.y, 0, 1, -1, 0))
        return false;
      for (int z = c.z0; z < c.z1; ++z) seen[(size_t)c.p + (size_t)L.c.plane * z] += 1;
    }
  for (int v : seen)
    if (v != 1) return false;
  return true;
}

static bool restriction(const Geo &g, int K) {
  mgd::MgLevel lv[kMaxLevels];
  if (mgd::level_shapes(g.nx, g.ny, g.nz, lv) < 2) return true;
  const mgd::MgLevel C = lv[1];
  mgd::RestrictMap M;
  const dim3 G = mgd::make_restrict_map(g, C, M, K ? (K > 1 ? K / 2 : 1) : 0);
  std::vector<int> wrote((size_t)C.N, 0), took((size_t)g.nx * g.ny * C.nz, 0);
  for (int bz = 0; bz < (int)G.z; ++bz)
    for (int by = 0; by < (int)G.y; ++by)
      for (int bx = 0; bx < (int)G.x; ++bx)
        for (int t = 0; t < 256; ++t) {
          const mgd::RestrictLane l = mgd::restrict_lane(M, t, bx, by, bz);
          if (l.x >= g.nx || l.y >= g.ny) continue;
          // partners of the shuffles: the same coarse node, the same planes
          const mgd::RestrictLane a = mgd::restrict_lane(M, (t & ~31) | ((t & 31) ^ 1), bx, by, bz);
          const mgd::RestrictLane b = mgd::restrict_lane(M, (t & ~31) | ((t & 31) ^ (1 << M.xl)), bx, by, bz);
          if (C.sx && (a.x != (l.x ^ 1) || a.y != l.y || a.Z0 != l.Z0)) return false;
          if (C.sy && (b.y != (l.y ^ 1) || b.x != l.x || b.Z0 != l.Z0)) return false;
          for (int Z = l.Z0; Z < l.Z0 + M.Kc && Z < C.nz; ++Z) {
            took[(size_t)l.x + (size_t)g.nx * (l.y + (size_t)g.ny * Z)] += 1;
            if (!(C.sx & l.lx & 1) && !(C.sy & l.ly & 1))
              wrote[(l.x >> C.sx) + (size_t)C.nx * ((l.y >> C.sy) + (size_t)C.ny * Z)] += 1;
          }
        }
  for (int v : wrote)
    if (v != 1) return false;
  for (int v : took)
    if (v != 1) return false;
  return true;
}

int main() {
  const int s[][3] = {{1, 1, 24},   {1, 1, 513},  {2, 1, 40},    {1, 3, 31},   {3, 5, 250},  {7, 9, 11},
                      {16, 16, 64}, {17, 15, 33}, {21, 19, 1},   {31, 2, 2},   {61, 47, 53}, {101, 97, 13},
                      {257, 3, 6},  {300, 40, 5}, {64, 64, 256}, {128, 128, 4}};
  for (const auto &v : s) {
    const Geo g{v[0], v[1], v[2], 1, 1, 1, (long long)v[0] * v[1] * v[2]};
    bool ok = true;
    for (int K = 0; K <= 16; ++K) ok = ok && columns(g, K) && restriction(g, K);
    std::printf("%dx%dx%d ok=%d\n", v[0], v[1], v[2], ok ? 1 : 0);
  }
  return 0;
}
