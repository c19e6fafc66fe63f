// Thread bodies of the Poisson solve's stencil kernels, shared by the single
// lattice (poisson.cu) and the batched form (batch.cu).  Pointers to values
// that another phase of the single-kernel solve writes (the vectors, the
// potential) carry no __restrict__: those must not become read-only-cache
// loads.
#pragma once

#include <type_traits>

#include "fp32_device.cuh"
#include "march.cuh"

namespace lbe {

// lap_mod(v)(r) at a fluid node, FP64.  With the link weights scaled by 6
// (2 nearest, 1 next-nearest, doubled towards solid unless dbl is false:
// the first-order rule) the sum needs one FP64 add per link:
// 6 lap = sum_i w_i v_i - (sum_i w_i) v0, w_i in {1, 2, 4}.
__device__ __forceinline__ double lap_at(const Offs &o, int r, uint32_t m, const double *v, bool dbl = true) {
  double s1 = 0.0, s2 = 0.0, s4 = 0.0;
  int wsum = 0;
#pragma unroll
  for (int i = 1; i < kQ; ++i) {
    const double vi = v[r + o.at(cx_of(i), cy_of(i), cz_of(i))];
    const int w = (c2_of(i) == 1 ? 2 : 1) * ((m & (1u << (i - 1))) || !dbl ? 1 : 2);
    if (w == 1) s1 += vi;
    else if (w == 2) s2 += vi;
    else s4 += vi;
    wsum += w;
  }
  return (s1 + 2.0 * s2 + 4.0 * s4 - (double)wsum * v[r]) * (1.0 / 6.0);
}

// Residual of the current potential; seeds the inner solve: r = (T)res,
// uj = r/diag (the CG's first update writes x, p and s).  max |res|/diag by
// atomicMax on its bits; the last block runs the outer test.
// MODE: R_N64 the FP64 form (FP64 potential and n); R_FX the FP32 form for
// a 1:1 salt: the fixed-point potential's Laplacian summed exactly in
// integers, the charge term from the fixed-point solute, both combined in
// float-float arithmetic; R_FXG the FP32 form for other salts (the exact
// Laplacian and the charge density in FP64); R_RHS a given rhs (linear
// solve A x = rhs with an FP64 iterate; its relative test also needs
// max |rhs|/diag); R_RHS_FF the same in float-float arithmetic (rhs values
// that are floats, x held as two floats).
// The potential of R_N64, R_FX and R_FXG is marched plane by plane
// (march.cuh) where a node's links all join fluid (their weights are then
// constants and integer sums do not depend on the order); a node next to a
// wall takes the per-link form.
enum { R_N64 = 0, R_FXG = 1, R_RHS = 2, R_FX = 3, R_RHS_FF = 4 };
struct ResArgs {
  Cols cols;
  Geo g;
  Phys P;
  P32 P3;
  const uint8_t *code;
  const uint32_t *mask;
  const double *n64;
  const int64_t *nq;
  const double *rhs;
  const double *phi;
  const float *phi_hi, *phi_lo;
  const int64_t *phifx;
  float c6_hi, c6_lo;
  int nblk, maxit, use_cond;
  PoissonCtl *c;
  double tol, tol_rel;
  cudaGraphConditionalHandle hout, hin;
};
template <int MODE>
constexpr bool kRhs = MODE == R_RHS || MODE == R_RHS_FF;
template <typename T, int MODE>
__device__ __forceinline__ void res_column(const ResArgs &A, const Column &c, T *r, T *uj, float &mx, float &mb) {
  constexpr bool MARCH = MODE == R_FX || MODE == R_FXG || MODE == R_N64;
  using V = typename std::conditional<MODE == R_N64, double, long long>::type;
  const V *v = MODE == R_N64 ? (const V *)A.phi : (const V *)A.phifx;
  const int plane = A.cols.plane, nz = A.cols.nz;
  ZMarch<V> m;
  if (MARCH) m.begin(v, c.o, c.p, plane, nz, c.z0);
#pragma unroll 1
  for (int z = c.z0; z < c.z1; ++z) {
    V v0 = 0, nsum = 0;
    int i = c.p + plane * z;
    if (A.cols.ahead && z + 1 + A.cols.ahead < c.z1) {
      const int j = i + plane * (1 + A.cols.ahead);
      if (MARCH) prefetch_l2(v + j);
      if (MODE == R_FX) {
        prefetch_l2(A.nq + j);
        prefetch_l2(A.nq + A.g.N + j);
      }
    }
    if (MARCH) nsum = m.step(v, c.o, c.p, plane, nz, z, v0, i);
    const int code = A.code[i];
    if (!code) {
      r[i] = uj[i] = (T)0;
      continue;
    }
    const bool wall = code & kCodeWall;
    const uint32_t mk = wall || !MARCH ? A.mask[i] : kLinkBits;
    T rt, dinv;
    if (MODE == R_FX || MODE == R_RHS_FF) {
      float S, E, B, Be;
      if (MODE == R_FX) {
        // 6 res = 6 lap + 6 (4 pi l_B s) (q+ - q-): 6 lap exact in fixed
        // point, split into float-float (the nearest float of the integer
        // sum and the float of its exact remainder), the charge term in
        // float-float too
        const long long L6 = wall ? fp32::lap6_fx_<false>(col_offs(c.o, plane, nz, z), i, mk, A.phifx)
                                  : (long long)(nsum - 24 * v0);
        const float Lh = fp32::ll2f(L6);
        const float Ll = fp32::ll2f(L6 - fp32::f2ll_rn(Lh));
        S = __fmul_rn(Lh, fp32::kPhiUnitF);
        E = __fmul_rn(Ll, fp32::kPhiUnitF);
        const long long dq = A.nq[i] - A.nq[A.g.N + i];
        const float dq_hi = fp32::ll2f(dq);
        const float dq_lo = fp32::ll2f(dq - fp32::f2ll_rn(dq_hi));  // exact remainder
        B = A.c6_hi * dq_hi;
        Be = fmaf(A.c6_hi, dq_hi, -B) + (A.c6_hi * dq_lo + A.c6_lo * dq_hi);  // product error and tails
      } else {
        // 6 res = 6 rhs + 6 lap(x), x = hi + lo, in float-float; rhs is a float
        if ((mk & kLinkBits) == kLinkBits)
          fp32::lap6_ff_<true>(col_offs(c.o, plane, nz, z), i, mk, A.phi_hi, A.phi_lo, S, E);
        else
          fp32::lap6_ff_<false>(col_offs(c.o, plane, nz, z), i, mk, A.phi_hi, A.phi_lo, S, E);
        const float bf = (float)A.rhs[i];
        B = 6.f * bf;
        Be = fmaf(6.f, bf, -B);  // 6 rhs = B + Be exactly
        mb = fmaxf(mb, finite_or_inf(fabsf(bf) * inv_diag<float>(code)));
      }
      float t, te;
      fp32::two_sum(S, B, t, te);
      rt = (T)((t + (te + (E + Be))) * (1.f / 6.f));
      dinv = inv_diag<T>(code);
    } else {
      double b;
      if (MODE == R_RHS) {
        b = A.rhs[i];
      } else {
        double q = 0.0;
        for (int k = 0; k < A.P.ns; ++k)
          q += A.P.z[k] * (MODE == R_FXG ? A.P3.rbd[k] + A.P3.sd[k] * (double)A.nq[k * A.g.N + i]
                                         : A.n64[k * A.g.N + i]);
        b = A.P.four_pi_lb * q;
      }
      double lap;
      if (MODE == R_FXG)
        lap = (double)(wall ? fp32::lap6_fx_<false>(col_offs(c.o, plane, nz, z), i, mk, A.phifx)
                            : (long long)(nsum - 24 * v0)) *
              (1.0 / 281474976710656.0 / 6.0);
      else if (MODE == R_N64 && !wall)
        lap = ((double)nsum - 24.0 * (double)v0) * (1.0 / 6.0);
      else
        lap = lap_at(col_offs(c.o, plane, nz, z), i, mk, A.phi, !(A.P.selfmask & kPlainLaplacian));
      const double rr = b + lap;
      rt = (T)rr;
      dinv = inv_diag<T>(code);
      if (MODE == R_RHS) mb = fmaxf(mb, finite_or_inf(fabsf((float)b) * (float)dinv));
    }
    r[i] = rt;
    uj[i] = rt * dinv;
    mx = fmaxf(mx, finite_or_inf(fabsf((float)rt) * (float)dinv));  // the stopping test needs no FP64
  }
}

// w = A u on a column chunk, and the chunk's part of (r,u) and (w,u)
template <typename T>
__device__ __forceinline__ void cg_b_column(const Cols &C, const Column &col, const uint8_t *code, const T *u, const T *r,
                                            T *w, T &ru, T &wu) {
  ZMarch<T> m;
  m.begin(u, col.o, col.p, C.plane, C.nz, col.z0);
  auto node = [&](int z) {
    T u0;
    int i;
    const T nsum = m.step(u, col.o, col.p, C.plane, C.nz, z, u0, i);
    const int cd = code[i];
    const T wv = cd ? ((T)((cd & kCodeDiag) + C.selfw) * u0 - nsum) * (T)(1.0 / 6.0) : (T)0;
    w[i] = wv;
    ru += r[i] * u0;
    wu += wv * u0;
  };
  // from HBM: prefetch, and several planes' loads in flight; from L2 a
  // short loop (on small lattices fetching unrolled code takes longer than
  // running it: FP64 solve of 4x4x64 0.78 against 0.94 ms per step)
  if (C.ahead) {
#pragma unroll 3
    for (int z = col.z0; z < col.z1; ++z) {
      if (z + 1 + C.ahead < col.z1) {
        prefetch_l2(u + m.j + C.plane * (1 + C.ahead));
        prefetch_l2(r + m.j + C.plane * C.ahead);
        prefetch_l2(code + m.j + C.plane * C.ahead);
      }
      node(z);
    }
  } else {
#pragma unroll 1
    for (int z = col.z0; z < col.z1; ++z) node(z);
  }
}
}  // namespace lbe
