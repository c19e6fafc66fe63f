// FP64 lattice kernels of one LBE time step (the "plain FP64" form).
//
//  * k_build_mask   per-node link mask of fluid neighbours (geometry set-up)
//  * k_init         uncharged capacitor, solvent at rest (Sec. "Potential and
//                   concentration profiles")
//  * k_sweep        fused ion link fluxes (Eq. LF1/LF2), solvent force from
//                   the link excess fluxes, D3Q19 BGK collision with Guo
//                   forcing (Eq. LBpop) and pull streaming with halfway
//                   bounce-back
//  * k_advect       cell-overlap advection of the solute by the velocity of
//                   the collision (scheme of Capuani et al., cited in the
//                   paper's Sec. "Lattice Boltzmann Electrokinetics")
//  * k_charge       induced electrode charge, Eq. Qelec
#include "lbe_internal.cuh"
#include "march.cuh"

namespace lbe {

namespace {

__device__ __forceinline__ long long nbr_i(const Geo &g, int x, int y, int z, int i) {
  return nbr(g, x, y, z, cx_of(i), cy_of(i), cz_of(i));
}

__global__ void k_build_mask(const Geo g, const uint8_t *__restrict__ id, uint32_t *__restrict__ mask) {
  long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  int x, y, z;
  coords(g, r, x, y, z);
  uint32_t m = id[r] == 0 ? kFluidBit : 0u;
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    long long r2 = nbr_i(g, x, y, z, i);
    if (r2 >= 0 && id[r2] == 0) m |= 1u << (i - 1);
  }
  for (int sz = -1; sz <= 1; sz += 2)
    for (int sy = -1; sy <= 1; sy += 2)
      for (int sx = -1; sx <= 1; sx += 2) {
        long long r2 = nbr(g, x, y, z, sx, sy, sz);
        if (r2 >= 0 && id[r2] == 0) m |= 1u << corner_bit(sx, sy, sz);
      }
  mask[r] = m;
}

// Node codes: 6 x the diagonal of -lap_mod (2 per nearest and 1 per
// next-nearest link, doubled towards solid except under the first-order rule,
// links of a node to itself left out), bit 7 for a node with a link to solid
__global__ void k_build_code(const Geo g, uint32_t selfmask, const uint32_t *__restrict__ mask,
                             uint8_t *__restrict__ code) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  const uint32_t m = mask[r];
  const int dbl = (selfmask & kPlainLaplacian) ? 1 : 2;
  int d = 0;
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    const uint32_t b = 1u << (i - 1);
    if (!(selfmask & b)) d += (c2_of(i) == 1 ? 2 : 1) * ((m & b) ? 1 : dbl);
  }
  code[r] = !(m & kFluidBit) ? 0 : (uint8_t)(d | ((m & kLinkBits) == kLinkBits ? 0 : kCodeWall));
}

__global__ void k_init(const Geo g, int ns, const uint8_t *__restrict__ id,
                       const double *psi, double *__restrict__ f, double *__restrict__ n,
                       double *__restrict__ phi, double *__restrict__ u, double rb0, double rb1,
                       double rb2, double rb3) {
  long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  const bool fl = id[r] == 0;
  const double rb[4] = {rb0, rb1, rb2, rb3};
#pragma unroll
  for (int i = 0; i < kQ; ++i) f[i * g.N + r] = fl ? w_of(i) : 0.0;
  for (int k = 0; k < ns; ++k) n[k * g.N + r] = fl ? rb[k] : 0.0;
  phi[r] = fl ? 0.0 : psi[id[r]];
  for (int a = 0; a < 3; ++a) u[a * g.N + r] = 0.0;
}

__global__ void k_init_phi(const Geo g, const uint8_t *__restrict__ id, const double *psi, double *__restrict__ phi) {
  long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  phi[r] = id[r] ? psi[id[r]] : 0.0;
}

__global__ void k_set_solid_phi(const Geo g, const uint8_t *__restrict__ id, const double *psi,
                                double *__restrict__ phi) {
  long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  if (id[r]) phi[r] = psi[id[r]];
}

// The two numbers of a link's potential step x from which its flux is formed.
// |x| < 1/4: sinh x and cosh x - 1, odd and even in x exactly, by Taylor series
// to x^7 and x^8 for |x| < 1/64 (most links: a kT/e over the Debye length), to
// x^11 and x^12 beyond, each truncated below 2e-17 relative.  Wide steps:
// expm1(-|x|) and expm1(|x|), out of line.  The ranges are tested on the high
// word, without the FP64 pipe.
struct LinkStep {
  double a, b;
  bool wide;
  int hi;  // high word of x
};
static __device__ __noinline__ double2 expm1_pm(double x) { return make_double2(expm1(-x), expm1(x)); }
__device__ __forceinline__ LinkStep link_step(double x) {
  LinkStep t;
  const int hi = __double2hiint(x) & 0x7fffffff;
  t.wide = hi >= 0x3fd00000;
  t.hi = __double2hiint(x);
  if (!t.wide) {
    const double x2 = x * x;
    double p = 1.0 / 5040.0, q = 1.0 / 40320.0;
    if (hi >= 0x3f900000) {
      p = fma(fma(1.0 / 39916800.0, x2, 1.0 / 362880.0), x2, p);
      q = fma(fma(1.0 / 479001600.0, x2, 1.0 / 3628800.0), x2, q);
    }
    p = fma(p, x2, 1.0 / 120.0);
    q = fma(q, x2, 1.0 / 720.0);
    p = fma(p, x2, 1.0 / 6.0);
    q = fma(q, x2, 1.0 / 24.0);
    p = fma(p, x2, 1.0);
    q = fma(q, x2, 0.5);
    t.a = p * x;
    t.b = q * x2;
  } else {
    const double2 w = expm1_pm(fabs(x));
    t.a = w.x;
    t.b = w.y;
  }
  return t;
}
// v with its sign bit flipped where `sign` has it set, on the integer pipe
constexpr int kSign = (int)0x80000000;
__device__ __forceinline__ double flip(double v, int sign) {
  return __hiloint2double(__double2hiint(v) ^ sign, __double2loint(v));
}
// A = n' (e^dmu - 1) - n (e^-dmu - 1) at dmu = x, or -x (neg: the sign bit).  A small step
// takes S sinh + D (cosh - 1), S = n + n', D = n' - n, whose terms do not cancel
// there; near equilibrium (n' = n e^-dmu) those two are e^|dmu| times as large
// as A, so that a wide step takes the exponentials themselves.  Both are one
// rounded product and one fused multiply-add, with the operands selected: no
// branch, and no FP64 instruction more for the small steps (sweep of 64x64x256
// 1.57 ms, as with sinh and cosh at every step; 1.64-1.67 with branches in
// line).  One expression for both signs: a copy for each made the code of a
// one-warp block so much longer to fetch that 4x4x64 took 42.8 us, 40.9 here.
// Wide steps: 2.98 ms, 3.09 with sinh and cosh formed from the exponentials.
// The rounded product is that of the growing exponential at either end of a
// link, so that its two ends get opposite values exactly.  (m0 = -n)
__device__ __forceinline__ double link_flux(const LinkStep &t, int neg, double n1, double m0, double S, double D) {
  const bool up = (t.hi ^ neg) >= 0;
  const double Sn = flip(S, neg);
  const double U = t.wide ? (up ? m0 : n1) : Sn, V = t.wide ? (up ? n1 : m0) : D;
  return fma(U, t.a, V * t.b);
}

// Link fluxes of Eq. LF2 and the solvent force.  With dmu = z (phi' - phi -
// E.c) and D = n' - n,
//   A = n' (e^{dmu} - 1) - n (e^{-dmu} - 1)     (small steps as S sinh + D (cosh - 1))
//   J = n' (1 + e^{dmu}) - n (1 + e^{-dmu}) = 2 D + A
// the flux is j = -d J/(2|c|) and the link excess flux g = j/d + D/|c| =
// -A/(2|c|) (D/|c| for an immobile species), summed into the force
// F = (1/(2 A0)) sum_i c_i sum_k g.  n* = n - sum_i j.  Every term is odd
// under reversal of the link, so its two ends move exactly opposite amounts.
// One series serves the species of valence +1 and -1.  Bound by the FP64
// pipe (1/64 of the FP32 rate): about 30 FP64 instructions per link of a 1:1
// salt with |dmu| < 1/4 against 80 with an exponential and two divisions per
// species.  J is exact to a few roundings of max(n, n') at any |dmu| near
// equilibrium (test_gpu_steep_links.py).  Axis and diagonal links are summed
// apart, so that 1/|c| multiplies once.
__device__ __forceinline__ void ion_fluxes(const Geo &g, const Phys &P, int r, const Offs &o, uint32_t m,
                                           const double *__restrict__ n, const double *__restrict__ phi,
                                           double *nstar_r, double F[3]) {
  const double phi0 = phi[r];
  double n0[LBE_MAX_SPECIES], acc1[LBE_MAX_SPECIES], acc2[LBE_MAX_SPECIES];
  // per species: valence +1, -1 or another, and immobile (whole-word tests of
  // the constants: a double comparison per link would run on the FP64 pipe)
  int kind[LBE_MAX_SPECIES];
  bool immobile[LBE_MAX_SPECIES];
#pragma unroll
  for (int k = 0; k < LBE_MAX_SPECIES; ++k) {
    n0[k] = k < P.ns ? n[k * g.N + r] : 0.0;
    acc1[k] = acc2[k] = 0.0;
    const int zh = __double2hiint(P.z[k]);
    kind[k] = zh == 0x3ff00000 ? 1 : (zh == (int)0xbff00000 ? -1 : 0);  // |z| is an integer below 5
    immobile[k] = __double_as_longlong(P.inv_d[k]) == 0;
  }
  double Fa[3] = {0.0, 0.0, 0.0}, Fd[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    if (!(m & (1u << (i - 1)))) continue;
    const int r2 = r + o.at(cx_of(i), cy_of(i), cz_of(i));
    const double x = phi[r2] - phi0 - P.e_dot_c[i];
    const LinkStep t = link_step(x);
    double gsum = 0.0;  // sum over species of -2 |c| g
#pragma unroll
    for (int k = 0; k < LBE_MAX_SPECIES; ++k) {
      if (k >= P.ns) break;
      const double n1 = n[k * g.N + r2];
      const double D = n1 - n0[k], S = n1 + n0[k];
      double A;
      const double m0 = flip(n0[k], kSign);
      if (kind[k] != 0) A = link_flux(t, kind[k] & kSign, n1, m0, S, D);
      else A = link_flux(link_step(P.z[k] * x), 0, n1, m0, S, D);
      const double J = fma(2.0, D, A);
      if (c2_of(i) == 1) acc1[k] += J;
      else acc2[k] += J;
      if (immobile[k]) A = -2.0 * D;
      gsum += A;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int ca = a == 0 ? cx_of(i) : (a == 1 ? cy_of(i) : cz_of(i));
      if (ca == 0) continue;
      double &f = c2_of(i) == 1 ? Fa[a] : Fd[a];
      f = ca > 0 ? f - gsum : f + gsum;
    }
  }
  constexpr double il = 0.70710678118654752440;  // 1/|c| of a diagonal link
#pragma unroll
  for (int k = 0; k < LBE_MAX_SPECIES; ++k)
    if (k < P.ns) nstar_r[k] = fma(0.5 * P.d[k], fma(il, acc2[k], acc1[k]), n0[k]);
#pragma unroll
  for (int a = 0; a < 3; ++a) F[a] = (0.5 * P.inv_2a0) * fma(il, Fd[a], Fa[a]);
}

// Pull streaming: population i at r comes from r - c_i = r + c_opp(i) if that
// node is fluid, else it is the population opp(i) that left r towards the
// wall and was bounced back (halfway bounce-back).
__device__ __forceinline__ void gather(const Geo &g, int r, const Offs &o, uint32_t m,
                                       const double *__restrict__ fin, double f[kQ]) {
  f[0] = fin[r];
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    const int io = opp_of(i);
    if (m & (1u << (io - 1)))
      f[i] = fin[i * g.N + (r + o.at(cx_of(io), cy_of(io), cz_of(io)))];
    else
      f[i] = fin[io * g.N + r];
  }
}

// Nodes of the FP64 sweep and advection: flattened, in blocks so small that
// even a lattice of a thousand nodes spreads over the SMs (their FP64 pipes
// bound both kernels: 4x4x64 in four blocks of 256 took 71 and 21 us).
struct FlatGeo {
  Geo g;
  FastDiv fx, fxy;
};
inline FlatGeo flat_geo(const Geo &g) {
  return FlatGeo{g, make_fastdiv((uint32_t)g.nx), make_fastdiv((uint32_t)((long long)g.nx * g.ny))};
}
inline unsigned flat_block(const Geo &g) { return g.N < 32768 ? 32 : 128; }
inline unsigned flat_grid(const Geo &g) { return (unsigned)((g.N + flat_block(g) - 1) / flat_block(g)); }
__device__ __forceinline__ bool flat_node(const FlatGeo &G, int &x, int &y, int &z, int &r) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= G.g.N) return false;
  r = (int)i;
  z = (int)fdiv(G.fxy, i);
  const int rem = r - z * (int)G.fxy.d;
  y = (int)fdiv(G.fx, (uint32_t)rem);
  x = rem - y * G.g.nx;
  return true;
}

// Fused step at a fluid node.  The collision takes the pairs c_i, -c_i
// together (even and odd parts of equilibrium and Guo source):
//   f'_i = (1 - omega) f_i + E_even +- E_odd,
//   E_even = w [omega rho (1 + 4.5 cu^2 - 1.5 uu) + guo (9 cu cF - 3 uF)]
//   E_odd  = w [3 omega rho cu + 3 guo cF]
// The kernel is bound by the FP64 pipe: on the 64x64x256 lattice 1.57 ms,
// against 3.14 ms with an exponential and divisions per link and species and
// one population at a time (4x4x64: 42 against 125 us).
template <bool FLOW>
__global__ void __launch_bounds__(128) k_sweep(const FlatGeo G, const Phys P, const uint32_t *__restrict__ mask,
                                               const double *__restrict__ fin, double *__restrict__ fout,
                                               const double *__restrict__ n, double *__restrict__ nstar,
                                               const double *__restrict__ phi, double *__restrict__ u) {
  const Geo &g = G.g;
  int x, y, z, r;
  if (!flat_node(G, x, y, z, r)) return;
  const uint32_t m = mask[r];
  if (!(m & kFluidBit)) return;
  const Offs o = offsets_of(g, x, y, z);
  double ns_r[LBE_MAX_SPECIES];
  double F[3];
  ion_fluxes(g, P, r, o, m, n, phi, ns_r, F);
#pragma unroll
  for (int k = 0; k < LBE_MAX_SPECIES; ++k)
    if (k < P.ns) nstar[k * g.N + r] = ns_r[k];
  if (!FLOW) return;

  double f[kQ];
  gather(g, r, o, m, fin, f);
  double rho = f[0], mx = 0.0, my = 0.0, mz = 0.0;
#pragma unroll
  for (int i = 1; i <= 9; ++i) {
    const double d = f[i] - f[i + 9];
    rho += f[i] + f[i + 9];
    if (cx_of(i)) mx += d;  // c_1..c_9 have c_x >= 0
    if (cy_of(i)) my = cy_of(i) > 0 ? my + d : my - d;
    if (cz_of(i)) mz = cz_of(i) > 0 ? mz + d : mz - d;
  }
  const double inv_rho = 1.0 / rho;
  const double ux = fma(0.5, F[0], mx) * inv_rho, uy = fma(0.5, F[1], my) * inv_rho,
               uz = fma(0.5, F[2], mz) * inv_rho;
  u[r] = ux;
  u[g.N + r] = uy;
  u[2 * g.N + r] = uz;
  const double uu = ux * ux + uy * uy + uz * uz;
  const double uF = ux * F[0] + uy * F[1] + uz * F[2];
  const double om = P.omega, gu = P.guo, keep = 1.0 - om;
  const double omr = om * rho;
  const double base = fma(omr, fma(-1.5, uu, 1.0), -3.0 * gu * uF);  // E_even / w at cu = cF = 0
  const double b2 = 4.5 * omr, d2 = 3.0 * omr, g3 = 3.0 * gu, g9 = 9.0 * gu;
  fout[r] = fma(keep, f[0], w_of(0) * base);
#pragma unroll
  for (int i = 1; i <= 9; ++i) {
    const double cu = cx_of(i) * ux + cy_of(i) * uy + cz_of(i) * uz;
    const double cF = cx_of(i) * F[0] + cy_of(i) * F[1] + cz_of(i) * F[2];
    const double ee = w_of(i) * fma(cu, fma(b2, cu, g9 * cF), base);
    const double eo = w_of(i) * fma(d2, cu, g3 * cF);
    const int io = i + 9;
    fout[i * g.N + r] = fma(keep, f[i], ee + eo);
    fout[io * g.N + r] = fma(keep, f[io], ee - eo);
  }
}

// Cell-overlap advection (pull form): node r collects, from every source
// q = r - s (s in {-1,0,1}^3) that is fluid, the share of q's solute whose
// displaced cell overlaps r; plus the shares of its own solute that would
// have landed on solid nodes.
__device__ __forceinline__ double ov(int s, double u) {
  return s == 0 ? 1.0 - fabs(u) : (s > 0 ? fmax(u, 0.0) : fmax(-u, 0.0));
}

__host__ __device__ constexpr int dir_bit(int dx, int dy, int dz) {
  // bit of the mask for the neighbour at offset (dx,dy,dz) != 0
  if (dx != 0 && dy != 0 && dz != 0) return corner_bit(dx, dy, dz);
  for (int i = 1; i < kQ; ++i)
    if (cx_of(i) == dx && cy_of(i) == dy && cz_of(i) == dz) return i - 1;
  return -1;
}

// the overlap at offset s can be nonzero: u has the sign of s (or s = 0); from
// the bits, without the FP64 pipe
__device__ __forceinline__ bool reaches(int s, double u) {
  return s == 0 || (s > 0 ? __double_as_longlong(u) > 0 : __double2hiint(u) < 0);
}

// A displaced cell only reaches the octant its velocity points to, so most
// sources are dismissed by the signs of their velocity before any FP64
// arithmetic (64x64x256: 0.32 ms, 0.49 when every overlap was evaluated).
__global__ void __launch_bounds__(128) k_advect(const FlatGeo G, int ns, const uint32_t *__restrict__ mask,
                                                const double *__restrict__ nin, const double *__restrict__ u,
                                                double *__restrict__ nout) {
  const Geo &g = G.g;
  int x, y, z, r;
  if (!flat_node(G, x, y, z, r)) return;
  const uint32_t m = mask[r];
  if (!(m & kFluidBit)) {
    for (int k = 0; k < ns; ++k) nout[k * g.N + r] = 0.0;
    return;
  }
  const Offs o = offsets_of(g, x, y, z);
  double acc[LBE_MAX_SPECIES] = {0.0, 0.0, 0.0, 0.0};
  const double ux = u[r], uy = u[g.N + r], uz = u[2 * g.N + r];
  double keep = 0.0;  // own shares bound for solid neighbours
#pragma unroll
  for (int d = 0; d < 27; ++d) {
    const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
    if (d == 13) {
      const double w = ov(0, ux) * ov(0, uy) * ov(0, uz);
#pragma unroll
      for (int k = 0; k < LBE_MAX_SPECIES; ++k)
        if (k < ns) acc[k] += w * nin[k * g.N + r];
      continue;
    }
    // source q = r - s exists as fluid iff the neighbour at -s is fluid
    if (m & (1u << dir_bit(-dx, -dy, -dz))) {
      const int q = r + o.at(-dx, -dy, -dz);
      const double vx = u[q], vy = u[g.N + q], vz = u[2 * g.N + q];
      if (reaches(dx, vx) && reaches(dy, vy) && reaches(dz, vz)) {
        const double w = ov(dx, vx) * ov(dy, vy) * ov(dz, vz);
#pragma unroll
        for (int k = 0; k < LBE_MAX_SPECIES; ++k)
          if (k < ns) acc[k] += w * nin[k * g.N + q];
      }
    }
    if (!(m & (1u << dir_bit(dx, dy, dz))) && reaches(dx, ux) && reaches(dy, uy) && reaches(dz, uz))
      keep += ov(dx, ux) * ov(dy, uy) * ov(dz, uz);
  }
#pragma unroll
  for (int k = 0; k < LBE_MAX_SPECIES; ++k)
    if (k < ns) nout[k * g.N + r] = acc[k] + keep * nin[k * g.N + r];
}

// Velocity and density of the current state, (sum f c + F/2)/rho with F from
// the current n and phi.
__global__ void k_moments(const Geo g, const Phys P, int flow, const uint32_t *__restrict__ mask,
                          const double *__restrict__ fin, const double *__restrict__ n,
                          const double *__restrict__ phi, double *__restrict__ rho_out,
                          double *__restrict__ u_out) {
  int x, y, z;
  long long r;
  if (!node_of(g, 1, 0, x, y, z, r)) return;
  const uint32_t m = mask[r];
  if (!(m & kFluidBit)) {
    if (rho_out) rho_out[r] = 0.0;
    if (u_out) u_out[r] = u_out[g.N + r] = u_out[2 * g.N + r] = 0.0;
    return;
  }
  const Offs o = offsets_of(g, x, y, z);
  double ns_r[LBE_MAX_SPECIES], F[3];
  ion_fluxes(g, P, (int)r, o, m, n, phi, ns_r, F);
  double f[kQ];
  gather(g, (int)r, o, m, fin, f);
  double rho = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
  for (int i = 0; i < kQ; ++i) {
    rho += f[i];
    mx += cx_of(i) * f[i];
    my += cy_of(i) * f[i];
    mz += cz_of(i) * f[i];
  }
  if (rho_out) rho_out[r] = rho;
  if (u_out) {
    u_out[r] = flow ? (mx + 0.5 * F[0]) / rho : 0.0;
    u_out[g.N + r] = flow ? (my + 0.5 * F[1]) / rho : 0.0;
    u_out[2 * g.N + r] = flow ? (mz + 0.5 * F[2]) / rho : 0.0;
  }
}

__global__ void k_gather_f(const Geo g, const uint32_t *__restrict__ mask, const double *__restrict__ fin,
                           double *__restrict__ out) {
  int x, y, z;
  long long r;
  if (!node_of(g, 1, 0, x, y, z, r)) return;
  const uint32_t m = mask[r];
  if (!(m & kFluidBit)) {
    for (int i = 0; i < kQ; ++i) out[i * g.N + r] = 0.0;
    return;
  }
  double f[kQ];
  gather(g, (int)r, offsets_of(g, x, y, z), m, fin, f);
  for (int i = 0; i < kQ; ++i) out[i * g.N + r] = f[i];
}

// Eq. Qelec, per block and electrode: -eps * sum over the block's electrode
// nodes of the modified Laplacian over links to fluid (factor 2 on every
// such boundary link).  Partials are summed in block order by k_charge_final.
__global__ void __launch_bounds__(kBlock) k_charge_partial(const Geo g, const Phys P, int n_elec,
                                                           const uint8_t *__restrict__ id,
                                                           const uint32_t *__restrict__ mask,
                                                           const double *__restrict__ phi,
                                                           double *__restrict__ part) {
  __shared__ double sh[kBlock / 32][LBE_MAX_ELECTRODES];
  double acc[LBE_MAX_ELECTRODES];
  for (int e = 0; e < n_elec; ++e) acc[e] = 0.0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < g.N;
       r += (long long)gridDim.x * blockDim.x) {
    const int e = id[r];
    if (!e) continue;
    const uint32_t m = mask[r];
    if (!(m & ((1u << 18) - 1))) continue;
    int x, y, z;
    coords(g, r, x, y, z);
    const double p0 = phi[r];
    double s = 0.0;
    for (int i = 1; i < kQ; ++i)
      if (m & (1u << (i - 1))) s += lapc_of(i) * P.solid_factor * (phi[nbr_i(g, x, y, z, i)] - p0);
    for (int k = 0; k < n_elec; ++k)
      if (k == e - 1) acc[k] += -P.eps * s;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int e = 0; e < n_elec; ++e) {
    double v = acc[e];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid][e] = v;
  }
  __syncthreads();
  if (threadIdx.x < n_elec) {
    double v = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) v += sh[w][threadIdx.x];
    part[(long long)blockIdx.x * n_elec + threadIdx.x] = v;
  }
}

__global__ void k_charge_final(int nblk, int n_elec, const double *__restrict__ part, double *__restrict__ q) {
  // one warp per electrode; lanes stride the partials, then a fixed tree
  const int e = blockIdx.x;
  if (e >= n_elec) return;
  double v = 0.0;
  for (int b = threadIdx.x; b < nblk; b += 32) v += part[(long long)b * n_elec + e];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (threadIdx.x == 0) q[e] = v;
}

// per-node term of Eq. Qelec (the map behind lbe_induced_charge)
__global__ void k_charge_node(const Geo g, const Phys P, const uint8_t *__restrict__ id,
                              const uint32_t *__restrict__ mask, const double *__restrict__ phi,
                              double *__restrict__ out) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= g.N) return;
  const uint32_t m = mask[r];
  if (!id[r] || !(m & ((1u << 18) - 1))) {
    out[r] = 0.0;
    return;
  }
  int x, y, z;
  coords(g, r, x, y, z);
  double s = 0.0;
  for (int i = 1; i < kQ; ++i)
    if (m & (1u << (i - 1))) s += lapc_of(i) * P.solid_factor * (phi[nbr_i(g, x, y, z, i)] - phi[r]);
  out[r] = -P.eps * s;
}

inline unsigned grid_for(long long N) { return (unsigned)((N + kBlock - 1) / kBlock); }
#define LAUNCH3(h) make_launch((h)->geo).grid, make_launch((h)->geo).block

}  // namespace

cudaError_t launch_build_mask(const Geo &g, const uint8_t *id, uint32_t *mask, cudaStream_t s) {
  k_build_mask<<<grid_for(g.N), kBlock, 0, s>>>(g, id, mask);
  return cudaGetLastError();
}

cudaError_t launch_build_code(const Geo &g, uint32_t selfmask, const uint32_t *mask, uint8_t *code, cudaStream_t s) {
  k_build_code<<<grid_for(g.N), kBlock, 0, s>>>(g, selfmask, mask, code);
  return cudaGetLastError();
}

// Electrode potentials are staged from a host stack array: an H2D copy from
// pageable memory returns only once the source has been consumed.
static cudaError_t stage_psi(lbe_handle *h) {
  double tmp[LBE_MAX_ELECTRODES + 1];
  tmp[0] = 0.0;
  for (int e = 0; e < h->n_elec; ++e) tmp[e + 1] = h->psi[e];
  return cudaMemcpyAsync(h->psi_dev, tmp, sizeof(double) * (h->n_elec + 1), cudaMemcpyHostToDevice,
                         h->stream);
}

cudaError_t launch_init_state(lbe_handle *h) {
  const double *rb = h->prm.rho_bulk;
  cudaError_t err = stage_psi(h);
  if (err != cudaSuccess) return err;
  k_init<<<grid_for(h->geo.N), kBlock, 0, h->stream>>>(h->geo, h->prm.nspecies, h->id, h->psi_dev,
                                                        h->f[h->cur], h->n, h->phi, h->u, rb[0], rb[1],
                                                        rb[2], rb[3]);
  return cudaGetLastError();
}

cudaError_t launch_init_phi(lbe_handle *h) {
  cudaError_t err = stage_psi(h);
  if (err != cudaSuccess) return err;
  k_init_phi<<<grid_for(h->geo.N), kBlock, 0, h->stream>>>(h->geo, h->id, h->psi_dev, h->phi);
  return cudaGetLastError();
}

cudaError_t launch_set_solid_phi(lbe_handle *h) {
  cudaError_t err = stage_psi(h);
  if (err != cudaSuccess) return err;
  k_set_solid_phi<<<grid_for(h->geo.N), kBlock, 0, h->stream>>>(h->geo, h->id, h->psi_dev, h->phi);
  return cudaGetLastError();
}

cudaError_t launch_sweep(lbe_handle *h) {
  const int nxt = h->cur ^ 1;
  const FlatGeo G = flat_geo(h->geo);
  (h->prm.flow ? k_sweep<true> : k_sweep<false>)<<<flat_grid(h->geo), flat_block(h->geo), 0, h->stream>>>(
      G, h->phys, h->mask, h->f[h->cur], h->f[nxt], h->n, h->nstar, h->phi, h->u);
  if (h->prm.flow) h->cur = nxt;
  return cudaGetLastError();
}

cudaError_t launch_advect(lbe_handle *h) {
  k_advect<<<flat_grid(h->geo), flat_block(h->geo), 0, h->stream>>>(flat_geo(h->geo), h->prm.nspecies, h->mask,
                                                                   h->nstar, h->u, h->n);
  return cudaGetLastError();
}

cudaError_t launch_moments(lbe_handle *h, double *rho_out, double *u_out) {
  k_moments<<<LAUNCH3(h), 0, h->stream>>>(h->geo, h->phys, h->prm.flow, h->mask,
                                                           h->f[h->cur], h->n, h->phi, rho_out, u_out);
  return cudaGetLastError();
}

cudaError_t launch_gather_f(lbe_handle *h, double *out) {
  k_gather_f<<<LAUNCH3(h), 0, h->stream>>>(h->geo, h->mask, h->f[h->cur], out);
  return cudaGetLastError();
}

cudaError_t launch_charge_node(lbe_handle *h, double *out) {
  k_charge_node<<<grid_for(h->geo.N), kBlock, 0, h->stream>>>(h->geo, h->phys, h->id, h->mask, h->phi, out);
  return cudaGetLastError();
}

cudaError_t launch_charge(lbe_handle *h) {
  k_charge_partial<<<h->qblk, kBlock, 0, h->stream>>>(h->geo, h->phys, h->n_elec, h->id, h->mask, h->phi,
                                                       h->qpart);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  k_charge_final<<<h->n_elec, 32, 0, h->stream>>>(h->qblk, h->n_elec, h->qpart, h->qout);
  return cudaGetLastError();
}

}  // namespace lbe
