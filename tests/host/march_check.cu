// Host check of the column-marching launch (march.cuh) and of the V-cycle's
// restriction map (vcycle.cuh): no GPU is used.  For ragged lattice shapes it
// walks every block and thread as the kernels do and checks that every node
// belongs to exactly one column chunk, that every coarse node's children lie
// in one group of lanes (written once), that the in-plane offsets name the
// periodic neighbours of nbr(), and that the number of chunks stays in the
// grid's limits.  The Python test parses the lines.
#include <cstdio>
#include <vector>

#include "../../paper_1907_04732_gb300/csrc/vcycle.cuh"

using namespace lbe;

static int wrapped(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

static bool check(int nx, int ny, int nz) {
  const Geo g{nx, ny, nz, 1, 1, 1, (long long)nx * ny * nz};
  const ColLaunch L = make_cols(g, 0u);
  if (L.block.x * L.block.y != 256 || L.grid.y > 65535u) return false;
  std::vector<int> seen((size_t)g.N, 0);
  for (unsigned by = 0; by < L.grid.y; ++by)
    for (unsigned bx = 0; bx < L.grid.x; ++bx)
      for (unsigned ty = 0; ty < L.block.y; ++ty)
        for (unsigned tx = 0; tx < L.block.x; ++tx) {
          const int p = (int)(bx * L.block.x + tx), z0 = (int)(by * L.block.y + ty) * L.c.K;
          if (p >= L.c.plane || z0 >= nz) continue;
          const int y = (int)fdiv(L.c.fnx, (uint32_t)p), x = p - y * nx;
          if (x < 0 || x >= nx || y != p / nx) return false;
          for (int z = z0; z < z0 + L.c.K && z < nz; ++z) seen[(size_t)p + (size_t)L.c.plane * z] += 1;
        }
  for (int v : seen)
    if (v != 1) return false;
  // the restriction into level 1
  mgd::MgLevel lv[kMaxLevels];
  if (mgd::level_shapes(nx, ny, nz, lv) < 2) return true;
  const mgd::MgLevel C = lv[1];
  mgd::RestrictMap M;
  const dim3 G = mgd::make_restrict_map(g, C, M);
  std::vector<int> wrote((size_t)C.N, 0), child((size_t)g.N, 0);
  for (int bz = 0; bz < (int)G.z; ++bz)
    for (int by = 0; by < (int)G.y; ++by)
      for (int bx = 0; bx < (int)G.x; ++bx)
        for (int t = 0; t < 256; ++t) {
          const int lane = t & 31, w = t >> 5;
          const int lx = lane & ((1 << M.xl) - 1), ly = (lane >> M.xl) & ((1 << M.yl) - 1), lz = lane >> (M.xl + M.yl);
          const int x = (bx << M.xl) + lx, y = ((by * M.wy + w % M.wy) << M.yl) + ly;
          const int Z0 = (((bz * (8 / M.wy) + w / M.wy) << M.zl) + lz) * M.Kc;
          if (x >= nx || y >= ny || Z0 >= C.nz) continue;
          for (int k = 0; k < M.Kc && Z0 + k < C.nz; ++k) {
            const int I = (x >> C.sx) + C.nx * ((y >> C.sy) + C.ny * (Z0 + k));
            if (!(C.sx & lx & 1) && !(C.sy & ly & 1)) wrote[I] += 1;
            for (int h = 0; h <= C.sz; ++h) {
              const int z = ((Z0 + k) << C.sz) + h;
              if (z < nz) child[(size_t)x + (size_t)nx * (y + (size_t)ny * z)] += 1;
            }
            // the shuffles' partners (lane ^ 1, lane ^ 2^xl) hold this node's siblings
            if (C.sx && (((bx << M.xl) + (lx ^ 1)) >> C.sx) != (x >> C.sx)) return false;
            if (C.sy && ((((by * M.wy + w % M.wy) << M.yl) + (ly ^ 1)) >> C.sy) != (y >> C.sy)) return false;
          }
        }
  for (int v : wrote)
    if (v != 1) return false;
  for (int v : child)
    if (v != 1) return false;
  // offsets of a plane's neighbours against the general neighbour function
  for (int y = 0; y < ny; ++y)
    for (int x = 0; x < nx; ++x) {
      const int xm = x == 0 ? nx - 1 : -1, xp = x == nx - 1 ? 1 - nx : 1;
      const int ym = y == 0 ? (ny - 1) * nx : -nx, yp = y == ny - 1 ? (1 - ny) * nx : nx;
      const int r = x + nx * y;
      if (r + xm != nbr(g, x, y, 0, -1, 0, 0) || r + xp != nbr(g, x, y, 0, 1, 0, 0) ||
          r + ym != nbr(g, x, y, 0, 0, -1, 0) || r + yp != nbr(g, x, y, 0, 0, 1, 0) ||
          r + xp + ym != wrapped(x + 1, nx) + nx * wrapped(y - 1, ny))
        return false;
    }
  return true;
}

int main() {
  const int s[][3] = {{1, 1, 24},  {1, 1, 513}, {2, 1, 40},   {1, 3, 31},    {3, 5, 250}, {7, 9, 11},     {16, 16, 64}, {17, 15, 33},
                      {21, 19, 1}, {31, 2, 2},  {61, 47, 53}, {101, 97, 13}, {128, 128, 4}, {257, 3, 6}, {300, 40, 5}, {64, 64, 256}};
  for (const auto &v : s) std::printf("%dx%dx%d ok=%d\n", v[0], v[1], v[2], check(v[0], v[1], v[2]) ? 1 : 0);
  // every divisor's remainders around its multiples, and the largest values
  bool ok = true;
  const uint32_t divs[] = {1, 2, 3, 5, 7, 61, 64, 101, 255, 256, 257, 4095, 65537, 1u << 30, 0x7fffffffu};
  for (uint32_t d : divs) {
    const FastDiv f = make_fastdiv(d);
    for (uint64_t k = 0; k < 5000; ++k)
      for (int o = -1; o <= 1; ++o) {
        const uint64_t n = k * d + o;
        if (n < 0x80000000ull && fdiv(f, (uint32_t)n) != (uint32_t)n / d) ok = false;
      }
    if (fdiv(f, 0x7fffffffu) != 0x7fffffffu / d) ok = false;
  }
  std::printf("fastdiv ok=%d\n", ok ? 1 : 0);
  return 0;
}
