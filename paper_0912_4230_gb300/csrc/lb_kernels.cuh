// Per-cell kernels of the GB300 lattice-Boltzmann library (templated on the
// population storage format, the permeability mode and the solute lattice).
//
// Layout: populations are structure-of-arrays, pop[q * N + n], n = x + nx*(y
// + ny*z), two buffers (A -> B -> A ...). Streaming is "pull": cell n reads
// f_q from n - c_q of the previous post-collision buffer, so every population
// is read once and written once per step and no atomics are needed. One
// thread owns one cell; consecutive threads are consecutive x, so each of the
// 19 loads and 19 stores of a warp is one contiguous 128-byte row segment
// (the x-shifted pulls straddle two segments, whose other half is read by the
// neighbouring warp and served from L1/L2).
#pragma once

#include <type_traits>

#include "lb_common.cuh"
#include "lb_ops.h"

namespace lbgb {

// Compile-time features of the per-cell step kernel, each a separate
// instantiation so that lattices without them keep the plain code:
// pressure / velocity faces of the fluid lattice, further solute species
// (1 .. S-1, advanced by the same thread after the fluid and species 0), and
// surface tension (A != 0; its terms would otherwise cost a predicated
// instruction or two per direction in every lattice).
enum : int { FEAT_OPEN = 1, FEAT_SPEC = 2, FEAT_TENS = 4 };

// the first direction of each pair of opposite directions (its partner is opp)
__host__ __device__ constexpr int pair_first(int k) {
  constexpr int t[9] = {1, 2, 5, 7, 8, 11, 13, 14, 17};
  return t[k];
}

template <int I, int N>
struct Unroll {
  template <class F>
  __device__ __forceinline__ static void run(F &&f) {
    f(std::integral_constant<int, I>{});
    Unroll<I + 1, N>::run(f);
  }
};
template <int N>
struct Unroll<N, N> {
  template <class F>
  __device__ __forceinline__ static void run(F &&) {}
};

// Additions and products that the compiler does not contract into an fma, so
// that every kernel forms the same values whatever surrounds them.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Values of the fluid and the solute lattice side by side. The collision
// does the same operations on f_q and h_q, so with FP32 collision the two
// share one packed instruction (fma / add / sub .rn.f32x2 of sm_100+, each
// half rounded as the scalar instruction): the step kernels are bound by
// instruction issue and load latency, and this halves the issue slots of the
// moments and the collision. FP64 has no packed form; without the solute
// lattice only f is there.
template <class Real, bool SOLUTE>
struct Lat {
  Real f, h;
  __device__ __forceinline__ static Lat mk(Real f, Real h) { return Lat{f, SOLUTE ? h : Real(0)}; }
  __device__ __forceinline__ Real lo() const { return f; }
  __device__ __forceinline__ Real hi() const { return SOLUTE ? h : Real(0); }
  __device__ __forceinline__ static Lat fma(Lat a, Lat b, Lat c) {
    return mk(::fma(a.f, b.f, c.f), SOLUTE ? ::fma(a.h, b.h, c.h) : Real(0));
  }
  __device__ __forceinline__ static Lat add(Lat a, Lat b) {
    return mk(add_rn(a.f, b.f), SOLUTE ? add_rn(a.h, b.h) : Real(0));
  }
  __device__ __forceinline__ static Lat sub(Lat a, Lat b) {
    return mk(sub_rn(a.f, b.f), SOLUTE ? sub_rn(a.h, b.h) : Real(0));
  }
  // gap = e.h - h/2, and the values af f + e.f, e.h - ah gap
  __device__ __forceinline__ static Lat relax(Lat v, Lat e, Real af, Real ah, Real &gap) {
    gap = SOLUTE ? ::fma(Real(-0.5), v.h, e.h) : Real(0);
    return mk(::fma(af, v.f, e.f), SOLUTE ? ::fma(-ah, gap, e.h) : Real(0));
  }
};
template <>
struct Lat<float, true> {
  unsigned long long v;
  __device__ __forceinline__ static Lat mk(float f, float h) {
    Lat r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(f), "f"(h));
    return r;
  }
  __device__ __forceinline__ float lo() const {
    float a;
    asm("{ .reg .f32 t; mov.b64 {%0, t}, %1; }" : "=f"(a) : "l"(v));
    return a;
  }
  __device__ __forceinline__ float hi() const {
    float b;
    asm("{ .reg .f32 t; mov.b64 {t, %0}, %1; }" : "=f"(b) : "l"(v));
    return b;
  }
  __device__ __forceinline__ static Lat fma(Lat a, Lat b, Lat c) {
    Lat r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
  }
  __device__ __forceinline__ static Lat add(Lat a, Lat b) {
    Lat r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
  }
  __device__ __forceinline__ static Lat sub(Lat a, Lat b) {
    Lat r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
  }
  __device__ __forceinline__ static Lat relax(Lat v, Lat e, float af, float ah, float &gap) {
    const Lat t = fma(mk(af, -0.5f), v, e);
    gap = t.hi();
    return mk(t.lo(), fmaf(-ah, gap, e.hi()));
  }
};

template <class Real>
__device__ __forceinline__ Real warp_sum(Real v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Geometry of one cell: wrapped index deltas to the six neighbours along the
// axes and the set of box faces the cell touches.
struct CellGeo {
  int dxm, dxp, dym, dyp, dzm, dzp;  // index delta to coord-1 / coord+1, wrapped
  unsigned onface;                   // faces_crossed bit layout
};

__device__ __forceinline__ CellGeo cell_geo_xyz(unsigned x, unsigned y, unsigned z, unsigned nx,
                                                unsigned ny, unsigned nz) {
  const int sy = int(nx), sz = int(nx * ny);
  CellGeo g;
  g.dxm = (x == 0) ? int(nx - 1) : -1;
  g.dxp = (x == nx - 1) ? -int(nx - 1) : 1;
  g.dym = (y == 0) ? int(ny - 1) * sy : -sy;
  g.dyp = (y == ny - 1) ? -int(ny - 1) * sy : sy;
  g.dzm = (z == 0) ? int(nz - 1) * sz : -sz;
  g.dzp = (z == nz - 1) ? -int(nz - 1) * sz : sz;
  g.onface = (x == 0 ? 1u : 0u) | (x == nx - 1 ? 2u : 0u) | (y == 0 ? 4u : 0u) |
             (y == ny - 1 ? 8u : 0u) | (z == 0 ? 16u : 0u) | (z == nz - 1 ? 32u : 0u);
  return g;
}

__device__ __forceinline__ CellGeo cell_geo(unsigned n, unsigned nx, unsigned ny, unsigned nz) {
  const unsigned x = n % nx, yz = n / nx, y = yz % ny, z = yz / ny;
  return cell_geo_xyz(x, y, z, nx, ny, nz);
}

// index delta of the pull source n - c_q (wrapped)
template <int q>
__device__ __forceinline__ int src_delta(const CellGeo &g) {
  return (cx(q) > 0 ? g.dxm : (cx(q) < 0 ? g.dxp : 0)) +
         (cy(q) > 0 ? g.dym : (cy(q) < 0 ? g.dyp : 0)) +
         (cz(q) > 0 ? g.dzm : (cz(q) < 0 ? g.dzp : 0));
}
// index delta of the neighbour n + c_q (wrapped)
template <int q>
__device__ __forceinline__ int ahead_delta(const CellGeo &g) {
  return src_delta<opp(q)>(g);
}

// Pull classes (shared by the step kernels and the debug export, which
// reports class c as -(1 + c)).
enum : int { PULL_CELL = 0, PULL_BOUNCE = 1, PULL_INLET = 2, PULL_OUTLET = 3,
             PULL_PRESSURE = 5, PULL_VELOCITY = 6 };

// Fluid class of population q: across a wall face or from a solid cell
// bounce-back; across a velocity face, else a pressure face, that face's
// rule (walls take precedence on edges, then velocity, then pressure).
template <int q>
__device__ __forceinline__ int fluid_class(const CellGeo &g, uint32_t link, unsigned f_wall) {
  if (q == 0) return PULL_CELL;
  const unsigned fc = faces_crossed(q) & g.onface;
  if (fc & f_wall) return PULL_BOUNCE;
  return ((link >> q) & 1u) ? PULL_BOUNCE : PULL_CELL;
}
template <int q>
__device__ __forceinline__ int fluid_class_open(const CellGeo &g, uint32_t link, unsigned f_wall,
                                                unsigned f_vel, unsigned f_press) {
  const unsigned fc = faces_crossed(q) & g.onface;
  if (q != 0 && !(fc & f_wall)) {
    if (fc & f_vel) return PULL_VELOCITY;
    if (fc & f_press) return PULL_PRESSURE;
  }
  return fluid_class<q>(g, link, f_wall);
}
// the face (2 axis + side) of kind `mask` that population q crosses first in
// axis order
template <int q>
__device__ __forceinline__ int crossed_face(const CellGeo &g, unsigned mask) {
  return __ffs(faces_crossed(q) & g.onface & mask) - 1;
}

template <int q>
__device__ __forceinline__ int solute_class(const CellGeo &g, uint32_t link, unsigned s_wall,
                                            unsigned s_inlet, unsigned s_outlet) {
  if (q == 0) return PULL_CELL;
  const unsigned fc = faces_crossed(q) & g.onface;
  if (fc & s_wall) return PULL_BOUNCE;
  if (fc & s_inlet) return PULL_INLET;
  if (fc & s_outlet) return PULL_OUTLET;
  return ((link >> q) & 1u) ? PULL_BOUNCE : PULL_CELL;
}

// Stream the fluid populations into d[] (f_q - w_q of the arriving populations).
// paired: 16-bit storage in the paired layout (rf then holds __half2 pairs).
template <class S>
__device__ __forceinline__ void gather_f(const typename S::T *__restrict__ fin, unsigned N,
                                         unsigned n, const CellGeo &g, uint32_t link,
                                         unsigned f_wall, typename S::Real (&d)[Q],
                                         const float *rf = nullptr, bool paired = false) {
  using Real = typename S::Real;
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const int cls = fluid_class<q>(g, link, f_wall);
    const long long src = (cls == PULL_BOUNCE) ? (long long)n : (long long)n + src_delta<q>(g);
    const size_t idx = (cls == PULL_BOUNCE) ? size_t(opp(q)) * N + n : size_t(q) * N + src;
    if constexpr (S::kShift) {
      if (paired)
        d[q] = wq<Real>(q) * (S::ld2(reinterpret_cast<const typename S::T2 *>(fin) + idx).x +
                              ld_ref2(rf + src).x);
      else
        d[q] = S::template ld_f<q>(fin + idx) + wq<Real>(q) * __ldg(rf + src);
    } else {
      d[q] = S::template ld_f<q>(fin + idx);
    }
  });
}

// Relaxation time from the viscosity law (Section 2, after Eq. eqsurftens;
// Eq. nuall for law 2 with t the step index after the increment).
template <class Real>
__device__ __forceinline__ Real tau_of(const StepArgs<Real> &a, Real C) {
  if (a.visc_law == 1) {
    const Real cl = C < Real(0) ? Real(0) : (C > Real(1) ? Real(1) : C);
    return a.tau0 + (a.tau1 - a.tau0) * cl;
  }
  if (a.visc_law == 2) {
    // nu_t = nu_g (1 + a e^{alpha t}), the same for every cell
    const Real nu = a.nu_t * exp(a.beta * (Real(1) - C));
    return Real(3) * nu + Real(0.5);
  }
  return a.tau;
}

// Viscosity from the law, not from the relaxation time: tau - 1/2 loses the
// leading digits of a rounded tau (2.4e-7 of nu at tau 0.6 in FP32, and as much of
// the velocity wherever the drag holds the flow).
template <class Real>
__device__ __forceinline__ Real nu_of(const StepArgs<Real> &a, Real C) {
  if (a.visc_law == 1) {
    const Real cl = C < Real(0) ? Real(0) : (C > Real(1) ? Real(1) : C);
    return fma(a.dnu, cl, a.nu0);
  }
  if (a.visc_law == 2) return a.nu_t * exp(a.beta * (Real(1) - C));
  return a.nu0;
}
// Both at once. In FP64 the two functions form the exponential of law 2 twice
// (90x90x1 wood sheet 26.7 us a step, 25.7 so). In FP32 they stay apart: together
// they change the order in which the compiler issues the cell's loads, 128^3
// Forchheimer 0.1065 to 0.1153 ms a step, three species 0.2126 to 0.2209.
template <class Real>
__device__ __forceinline__ void tau_nu(const StepArgs<Real> &a, Real C, Real &tau, Real &nu) {
  if constexpr (sizeof(Real) == 4) {
    tau = tau_of(a, C);
    nu = nu_of(a, C);
  } else {
    tau = a.tau;
    nu = a.nu0;
    if (a.visc_law == 1) {
      const Real cl = C < Real(0) ? Real(0) : (C > Real(1) ? Real(1) : C);
      tau = a.tau0 + (a.tau1 - a.tau0) * cl;
      nu = fma(a.dnu, cl, a.nu0);
    } else if (a.visc_law == 2) {
      nu = a.nu_t * exp(a.beta * (Real(1) - C));
      tau = Real(3) * nu + Real(0.5);
    }
  }
}

// c_q . (a0, a1, a2) by additions of the axes that q has (a product with a zero
// component is an instruction the compiler may not drop; in FP64 it holds the
// pipe for 64 cycles).
template <int q, class Real>
__device__ __forceinline__ Real dot_c(Real a0, Real a1, Real a2) {
  if constexpr (cx(q) != 0) {
    const Real s = cx(q) > 0 ? a0 : -a0;
    if constexpr (cy(q) != 0) return cy(q) > 0 ? add_rn(s, a1) : sub_rn(s, a1);
    if constexpr (cz(q) != 0) return cz(q) > 0 ? add_rn(s, a2) : sub_rn(s, a2);
    return s;
  } else if constexpr (cy(q) != 0) {
    const Real s = cy(q) > 0 ? a1 : -a1;
    if constexpr (cz(q) != 0) return cz(q) > 0 ? add_rn(s, a2) : sub_rn(s, a2);
    return s;
  } else if constexpr (cz(q) != 0) {
    return cz(q) > 0 ? a2 : -a2;
  } else {
    return Real(0);
  }
}

// Reciprocal in the collision type: one correctly rounded reciprocal
// instruction sequence in FP32, exact division in FP64.
__device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }

// Reciprocal of a normal number below 2^126 (density, porosity, relaxation time,
// 1 + drag, a determinant below 2^120; beyond, the approximation is flushed to 0
// and the correction of an infinity is not a number): the hardware's approximation
// and a Newton-Raphson step, r <- r + r e, e = 1 - x r, in FP32 (from 1 ulp) or the
// third-order step r + r (e + e^2) in FP64 (from 2^-20 to beyond 2^-53), without
// the range checks and slow path of the exact reciprocal. FP32 results are those of
// the correctly rounded reciprocal for every argument from 2^-100 to 2^126; of
// 1.3e9 random FP64 ones 0.03 % differ in the last bit. An FP64 instruction holds its
// pipe for 64 cycles a warp on this chip (measured, whatever the active lanes), so 3
// instead of ~10 count there.
__device__ __forceinline__ float rcp1(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double rcp1(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Inside an iteration that corrects its own errors (the Forchheimer Newton
// solve) FP32 takes the hardware's single-instruction approximations (at
// most 1 ulp off: PTX rcp.approx / sqrt.approx); FP64 keeps exact operations.
__device__ __forceinline__ float rcp_iter(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double rcp_iter(double x) { return 1.0 / x; }
__device__ __forceinline__ float sqrt_iter(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double sqrt_iter(double x) { return sqrt(x); }

// Lambda V' = r, Lambda = 1 + hs K^-1, where the determinant leaves the range of
// FP32 (nearly tight cells, K below ~1e-13 in every direction): with S = diag(s_i),
// s_i the power of two that brings s_i^2 l_ii into [1, 4), V' = S (S Lambda S)^-1
// S r, whose determinant is at most 64. Scaling by powers of two rounds nothing.
// again(i) loads row i of K^-1 anew: kept in registers for this rare branch, the
// rows cost a 256^3 FP16 solve 1.8 % in spills (25.50 to 25.95 ms; 25.76 so).
template <class Real, class KV>
__device__ __forceinline__ void tight_solve(KV again, Real hs, Real r0, Real r1, Real r2,
                                            Real (&Vp)[3]) {
  const auto half_scale = [](Real l) { return scalbn(Real(1), -(ilogb(l) / 2)); };
  Real l00 = Real(1) + hs * again(0), l11 = Real(1) + hs * again(1), l22 = Real(1) + hs * again(2);
  const Real s0 = half_scale(l00), s1 = half_scale(l11), s2 = half_scale(l22);
  l00 = l00 * s0 * s0;
  l11 = l11 * s1 * s1;
  l22 = l22 * s2 * s2;
  const Real l01 = hs * again(3) * s0 * s1, l12 = hs * again(4) * s1 * s2,
             l02 = hs * again(5) * s0 * s2;
  r0 *= s0;
  r1 *= s1;
  r2 *= s2;
  const Real c00 = l11 * l22 - l12 * l12, c01 = l02 * l12 - l01 * l22, c02 = l01 * l12 - l02 * l11;
  const Real c11 = l00 * l22 - l02 * l02, c12 = l01 * l02 - l00 * l12, c22 = l00 * l11 - l01 * l01;
  const Real idet = Real(1) / (l00 * c00 + l01 * c01 + l02 * c02);
  Vp[0] = s0 * ((c00 * r0 + c01 * r1 + c02 * r2) * idet);
  Vp[1] = s1 * ((c01 * r0 + c11 * r1 + c12 * r2) * idet);
  Vp[2] = s2 * ((c02 * r0 + c12 * r1 + c22 * r2) * idet);
}

// V' = Lambda^-1 (V + eps G / 2), Lambda = I + (eps nu / 2) K^-1, and
// F^ext = -eps nu K^-1 V' + eps G (Eqs. forcement, expandV, expandVsub).
// kv(r) returns row r of the cell's K^-1 (diagonal: xx, yy, zz; full: xx, yy,
// zz, xy, yz, zx); again(r) loads it anew, and as row 6 the porosity.
//
// KM_FORCH adds the Forchheimer drag of the porous-flow model the paper builds
// on (the paper names the term without an equation): F^ext = -eps nu K^-1 V'
// - eps F_eps |V'| K^-1/2 V' + eps G, F_eps = cF 1.75 / sqrt(150 eps^3), for a
// diagonal K. With V' = V + F^ext/2, V'_i = r_i / (a_i + b_i s), r = V + eps
// G/2, a_i = 1 + eps nu k_i / 2, b_i = eps F_eps sqrt(k_i) / 2, where s = |V'|
// is the root of phi(s) = s - |V'(s)|. Newton's method on phi from the
// closed form of an isotropic medium with the r^2-weighted a and b; three
// iterations in FP32 and four in FP64 reach the root to rounding for K from
// 1e-4 to 1e2, 100:1 anisotropy and cF up to 20.
template <int KMODE, bool EXACT = false, class Real, class KV, class KA>
__device__ __forceinline__ void velocity_solve_kv(KV kv, KA again, Real eps, Real nu, const Real (&V)[3],
                                                  const Real (&G)[3], Real cF, Real (&Vp)[3],
                                                  Real (&Fe)[3]) {
  const Real r0 = V[0] + Real(0.5) * eps * G[0];
  const Real r1 = V[1] + Real(0.5) * eps * G[1];
  const Real r2 = V[2] + Real(0.5) * eps * G[2];
  const Real en = eps * nu;
  if (KMODE == KM_NONE) {
    Vp[0] = r0; Vp[1] = r1; Vp[2] = r2;
    Fe[0] = eps * G[0]; Fe[1] = eps * G[1]; Fe[2] = eps * G[2];
  } else if (KMODE == KM_FORCH) {
    const Real k[3] = {kv(0), kv(1), kv(2)};
    const Real r[3] = {r0, r1, r2};
    const Real Fer = cF * Real(1.75) * rcp(sqrt(Real(150) * eps * eps * eps));
    const Real hs = Real(0.5) * en, hc = Real(0.5) * eps * Fer;
    Real a[3], b[3], d[3];
    for (int i = 0; i < 3; ++i) {
      d[i] = sqrt(k[i]);
      a[i] = Real(1) + hs * k[i];
      b[i] = hc * d[i];
    }
    const Real ws = r0 * r0 + r1 * r1 + r2 * r2;
    Real s = Real(0);
    if (ws > Real(0)) {
      const Real iws = rcp(ws);
      const Real ab = (r0 * r0 * a[0] + r1 * r1 * a[1] + r2 * r2 * a[2]) * iws;
      const Real bb = (r0 * r0 * b[0] + r1 * r1 * b[1] + r2 * r2 * b[2]) * iws;
      const Real rn = sqrt(ws);
      s = Real(2) * rn * rcp_iter(ab + sqrt_iter(ab * ab + Real(4) * bb * rn));
      // Newton on phi(s) = s - |V'(s)|: s <- s - (s - |V'|) |V'| / (|V'| + g),
      // g = sum_i V'_i^2 b_i / (a_i + b_i s); the iteration absorbs the
      // approximate reciprocals and roots, the final V' takes exact ones
      constexpr int kIters = sizeof(Real) == 4 ? 3 : 4;
      for (int it = 0; it < kIters; ++it) {
        Real vv = Real(0), g = Real(0);
        for (int i = 0; i < 3; ++i) {
          const Real iD = rcp_iter(a[i] + b[i] * s), v = r[i] * iD;
          vv += v * v;
          g += v * v * b[i] * iD;
        }
        const Real vn = sqrt_iter(vv);
        s -= (s - vn) * vn * rcp_iter(vn + g);
      }
    }
    for (int i = 0; i < 3; ++i) Vp[i] = r[i] * rcp(a[i] + b[i] * s);
    const Real sp = sqrt(Vp[0] * Vp[0] + Vp[1] * Vp[1] + Vp[2] * Vp[2]);
    for (int i = 0; i < 3; ++i) Fe[i] = -(en * k[i] + eps * Fer * d[i] * sp) * Vp[i] + eps * G[i];
  } else if (KMODE == KM_DIAG) {
    const Real kx = kv(0), ky = kv(1), kz = kv(2);
    const Real hs = Real(0.5) * en;
    if constexpr (sizeof(Real) == 8) {
      // one reciprocal for the three (k <= 1e45, so the product is finite)
      const Real e0 = en * kx, e1 = en * ky, e2 = en * kz;
      const Real lx = fma(Real(0.5), e0, Real(1)), ly = fma(Real(0.5), e1, Real(1)),
                 lz = fma(Real(0.5), e2, Real(1));
      const Real lxy = lx * ly, i3 = rcp1(lxy * lz), iz = i3 * lz;
      Vp[0] = r0 * (iz * ly);
      Vp[1] = r1 * (iz * lx);
      Vp[2] = r2 * (i3 * lxy);
      Fe[0] = fma(-e0, Vp[0], eps * G[0]);
      Fe[1] = fma(-e1, Vp[1], eps * G[1]);
      Fe[2] = fma(-e2, Vp[2], eps * G[2]);
      return;
    }
    const Real lx = Real(1) + hs * kx, ly = Real(1) + hs * ky, lz = Real(1) + hs * kz;
    if constexpr (EXACT) {
      Vp[0] = r0 * rcp(lx);
      Vp[1] = r1 * rcp(ly);
      Vp[2] = r2 * rcp(lz);
    } else {
      Vp[0] = r0 * rcp1(lx);
      Vp[1] = r1 * rcp1(ly);
      Vp[2] = r2 * rcp1(lz);
    }
    Fe[0] = -en * kx * Vp[0] + eps * G[0];
    Fe[1] = -en * ky * Vp[1] + eps * G[1];
    Fe[2] = -en * kz * Vp[2] + eps * G[2];
  } else {
    const Real kxx = kv(0), kyy = kv(1), kzz = kv(2);
    const Real kxy = kv(3), kyz = kv(4), kzx = kv(5);
    const Real hs = Real(0.5) * en;
    const Real l00 = Real(1) + hs * kxx, l11 = Real(1) + hs * kyy, l22 = Real(1) + hs * kzz;
    const Real l01 = hs * kxy, l12 = hs * kyz, l02 = hs * kzx;
    // adjugate of the symmetric matrix Lambda
    const Real c00 = l11 * l22 - l12 * l12, c01 = l02 * l12 - l01 * l22, c02 = l01 * l12 - l02 * l11;
    const Real c11 = l00 * l22 - l02 * l02, c12 = l01 * l02 - l00 * l12, c22 = l00 * l11 - l01 * l01;
    const Real det = l00 * c00 + l01 * c01 + l02 * c02;
    const Real idet = EXACT ? Real(1) / det : rcp1(det);
    Vp[0] = (c00 * r0 + c01 * r1 + c02 * r2) * idet;
    Vp[1] = (c01 * r0 + c11 * r1 + c12 * r2) * idet;
    Vp[2] = (c02 * r0 + c12 * r1 + c22 * r2) * idet;
    Fe[0] = -en * (kxx * Vp[0] + kxy * Vp[1] + kzx * Vp[2]) + eps * G[0];
    Fe[1] = -en * (kxy * Vp[0] + kyy * Vp[1] + kyz * Vp[2]) + eps * G[1];
    Fe[2] = -en * (kzx * Vp[0] + kyz * Vp[1] + kzz * Vp[2]) + eps * G[2];
    // Lambda >= 1, so det bounds every cofactor; a sum that overflows may end at
    // either infinity or not a number. (FP64 stays in range: k <= 1e45.)
    if (sizeof(Real) == 4 && !(fabs(det) < Real(0x1p120))) {
      // V' = V + F^ext / 2 = r + (F^ext - eps G) / 2. (A product shared with the
      // lines above would change which of their operations the compiler fuses,
      // so eps is loaded too.)
      tight_solve(again, hs, r0, r1, r2, Vp);
      const Real e = again(6);
      Fe[0] = Real(2) * (Vp[0] - r0) + e * G[0];
      Fe[1] = Real(2) * (Vp[1] - r1) + e * G[1];
      Fe[2] = Real(2) * (Vp[2] - r2) + e * G[2];
    }
  }
}

template <int KMODE, class Real>
__device__ __forceinline__ void velocity_solve(const Real *__restrict__ kinv, unsigned N,
                                               unsigned n, Real eps, Real nu, const Real (&V)[3],
                                               const Real (&G)[3], Real (&Vp)[3],
                                               Real (&Fe)[3]) {
  auto row = [&](int r) { return r < 6 ? __ldg(kinv + size_t(r) * N + n) : eps; };
  velocity_solve_kv<KMODE>(row, row, eps, nu, V, G, Real(0), Vp, Fe);
}

// Colour gradient F = sum_q rhohat(x + c_q) c_q (Eq. macros); a step out
// through a wall face sees wall_rho (solid cells already hold wall_rho).
template <class Real>
__device__ __forceinline__ void colour_gradient(const Real *__restrict__ rh, unsigned n,
                                                const CellGeo &g, unsigned f_wall, Real wall_rho,
                                                Real (&F)[3]) {
  F[0] = F[1] = F[2] = Real(0);
  Unroll<1, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const bool out = (faces_ahead(q) & g.onface & f_wall) != 0;
    const Real r = out ? wall_rho : __ldg(rh + (long long)n + ahead_delta<q>(g));
    if (cx(q)) F[0] += Real(cx(q)) * r;
    if (cy(q)) F[1] += Real(cy(q)) * r;
    if (cz(q)) F[2] += Real(cz(q)) * r;
  });
}

// BGK collision with the porous equilibrium (Eqs. equilc1, equilc2) and the
// forcing terms (Eq. coeffforce1, with the weight and density factor w_q rho)
// for one direction, in deviation form:
//   f~_q - w_q = (f_q - w_q)(1 - 1/tau) + (f^eq_q - w_q)/tau + T_q.
// fold() gathers the per-cell factors of the last two terms, so that per
// direction they are w_q b_q with
//   b_q = K + cu (B3 + B45 cu + P9 cF) + P3 cF [+ S2 (c_q.F)^2],
// cu = c_q.V', cF = c_q.F_e (K0 in place of K for the rest direction), taken
// as scale (b_q - shift). Used by the initialisation (feq_dev), the
// free surface and 16-bit storage; the FP32/FP64 porous step folds further
// (collide_tail).
template <class Real>
struct FluidCollide {
  Real drho, rho, ie, uu, uF, itau, omt, pre, stc, Fn, iFn;
  Real Vp[3], Fe[3], F[3];
  bool st;
  Real K, K0, B3, B45, P9, P3, S2;

  __device__ __forceinline__ void fold(Real scale, Real shift) {
    // 1/tau (f^eq - w) + T at cu = cF = 0, without the surface-tension part
    const Real kb = itau * drho - Real(1.5) * itau * rho * ie * uu - Real(3) * pre * ie * uF;
    const Real ks = st ? itau * stc * Fn : Real(0);
    K = scale * (kb - ks - shift);
    K0 = scale * (kb + ks - shift);
    B3 = scale * Real(3) * itau * rho;
    B45 = scale * Real(4.5) * itau * rho * ie;
    P9 = scale * Real(9) * pre * ie;
    P3 = scale * Real(3) * pre;
    S2 = st ? scale * itau * stc * iFn : Real(0);
  }
  template <int q>
  __device__ __forceinline__ Real br() const {
    if (q == 0) return K0;
    const Real cu = dot_c<q>(Vp[0], Vp[1], Vp[2]);
    const Real cF = dot_c<q>(Fe[0], Fe[1], Fe[2]);
    Real b = cu * (B3 + B45 * cu + P9 * cF) + (P3 * cF + K);
    if (st) {
      const Real cs = dot_c<q>(F[0], F[1], F[2]);
      b += S2 * cs * cs;
    }
    return b;
  }
  // Even and odd part of b_q for a pair of opposite directions: K + cu (B45 cu
  // + P9 cF) [+ S2 (c.F)^2] and B3 cu + P3 cF (cu = c_q.V', cF = c_q.F_e)
  template <int q>
  __device__ __forceinline__ void even_odd(Real cu, Real &ev, Real &od) const {
    const Real cF = Real(cx(q)) * Fe[0] + Real(cy(q)) * Fe[1] + Real(cz(q)) * Fe[2];
    ev = fma(cu, fma(B45, cu, P9 * cF), K);
    if (st) {
      const Real cs = dot_c<q>(F[0], F[1], F[2]);
      ev = fma(S2 * cs, cs, ev);
    }
    od = fma(B3, cu, P3 * cF);
  }
  // f^eq_q - w_q (with the surface-tension part), for initialisation
  template <int q>
  __device__ __forceinline__ Real feq_dev() const {
    constexpr Real w = wq<Real>(q);
    if (q == 0) return w * (drho - rho * Real(1.5) * ie * uu) + (st ? stc * w * Fn : Real(0));
    const Real cu = dot_c<q>(Vp[0], Vp[1], Vp[2]);
    Real e = w * (drho + rho * (Real(3) * cu + Real(4.5) * ie * cu * cu - Real(1.5) * ie * uu));
    if (st) {
      const Real cs = dot_c<q>(F[0], F[1], F[2]);
      e += w * stc * (cs * cs * iFn - Fn);
    }
    return e;
  }
  // f~_q - w_q after fold(1, 0)
  template <int q>
  __device__ __forceinline__ Real post(Real d) const {
    return fma(wq<Real>(q), br<q>(), d * omt);
  }
};

// Exported fields, 6 x N floats: rho [N], u packed per cell [3N], C [N], nu [N].
template <class Real>
__device__ __forceinline__ void write_fields(float *fl, unsigned N, unsigned n, Real rho,
                                             const Real (&u)[3], Real C, Real nu) {
  fl[n] = float(rho);
  fl[size_t(N) + 3 * size_t(n)] = float(u[0]);
  fl[size_t(N) + 3 * size_t(n) + 1] = float(u[1]);
  fl[size_t(N) + 3 * size_t(n) + 2] = float(u[2]);
  fl[4 * size_t(N) + n] = float(C);
  fl[5 * size_t(N) + n] = float(nu);
}

__device__ __forceinline__ void zero_fields(float *fl, unsigned N, unsigned n) {
  fl[n] = 0.0f;
  fl[size_t(N) + 3 * size_t(n)] = 0.0f;
  fl[size_t(N) + 3 * size_t(n) + 1] = 0.0f;
  fl[size_t(N) + 3 * size_t(n) + 2] = 0.0f;
  fl[4 * size_t(N) + n] = 0.0f;
  fl[5 * size_t(N) + n] = 0.0f;
}

template <class Real>
__device__ __forceinline__ Real st_threshold();
template <>
__device__ __forceinline__ float st_threshold<float>() { return 1e-20f; }
template <>
__device__ __forceinline__ double st_threshold<double>() { return 1e-30; }

// Flags a warp whose mass or solute sum is not finite. The sums themselves
// (10 shuffles and additions of each) are only formed when some lane's value
// is large or not a number; below 1e36 the sum of 32 is finite.
template <class Real>
__device__ __forceinline__ void finite_check(DevState *state, Real drho, Real sC) {
  // (FP64: by the high words, on the integer pipe; the FP64 one is the
  // bottleneck of those kernels)
  bool fine;
  if constexpr (sizeof(Real) == 8)
    fine = (__double2hiint(drho) & 0x7fffffff) < 0x47700000 &&
           (__double2hiint(sC) & 0x7fffffff) < 0x47700000;
  else
    fine = fabs(drho) < Real(1e36) && fabs(sC) < Real(1e36);
  if (__any_sync(0xffffffffu, !fine)) {
    const Real m = warp_sum(drho), c = warp_sum(sC);
    if ((threadIdx.x & 31u) == 0 && !(isfinite(m) && isfinite(c))) atomicOr(&state->status, 1u);
  }
}

// Per-warp FP64 reductions of a step. Solute fluxes through inlet/outlet
// faces are accumulated into one FP64 slot pair per warp of the launch
// (each warp owns its slots across steps, so the running sums are
// deterministic; lb_reduce adds the slots in a fixed order). On checked
// steps the warp's mass and solute sums are tested for NaN/Inf.
template <class Real>
__device__ __forceinline__ void warp_reductions(const StepArgs<Real> &a, unsigned warp_gid,
                                                bool open_face, Real fin, Real fout, Real drho,
                                                Real sC) {
  const unsigned lane = threadIdx.x & 31u;
  if (a.flux && __any_sync(0xffffffffu, open_face)) {
    const Real si = warp_sum(fin), so = warp_sum(fout);
    if (lane == 0) {
      a.flux_slots[2 * size_t(warp_gid)] += double(si);
      a.flux_slots[2 * size_t(warp_gid) + 1] += double(so);
    }
  }
  if (a.reduce) finite_check(a.state, drho, sC);
}

// Reciprocals up to the velocity: with 16-bit storage the correctly rounded
// one. In a tight medium the drag balances the body force, F_e is the small
// difference of the two, and its FP32 rounding is as large as the last bit of
// a 16-bit remainder.
template <class S>
__device__ __forceinline__ typename S::Real rcp_as(typename S::Real x) {
  if constexpr (S::kShift)
    return rcp(x);
  else
    return rcp1(x);
}

// Moments of the arriving populations: drho = sum_q (f_q - w_q), V = j / rho
// with j = sum_q c_q (f_q - w_q), rho = 1 + drho, and the solute total sC =
// sum_q h_q. FP32 / FP64 storage takes opposite directions together: their
// sums feed drho and sC, their differences j, and both are kept in sd for
// the collision (sd[k] the sum and sd[9 + k] the difference of pair k, sd[18]
// the rest direction). 16-bit storage gives the values per unit weight, e_q =
// (f_q - w_q)/w_q and h_q/w_q, and sums them with their weights in the order
// of q (sd unused): two roundings that differ in one bit end in different
// 16-bit remainders.
template <class S, bool SOLUTE, class FV, class HV>
__device__ __forceinline__ void moments(FV fv, HV hv, typename S::Real &drho,
                                        typename S::Real &sC, typename S::Real (&V)[3],
                                        Lat<typename S::Real, SOLUTE> (&sd)[Q]) {
  using Real = typename S::Real;
  using L = Lat<Real, SOLUTE>;
  auto in = [&](auto qc) { return L::mk(fv(qc), hv(qc)); };
  L tot = L::mk(Real(0), Real(0)), axis = tot;
  Real jd[3] = {Real(0), Real(0), Real(0)}, ja[3] = {Real(0), Real(0), Real(0)};
  if constexpr (S::kShift) {
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      constexpr Real w = wq<Real>(q);
      tot = L::fma(L::mk(w, w), in(qc), tot);
      if (cx(q)) jd[0] = fma(Real(cx(q)) * w, fv(qc), jd[0]);
      if (cy(q)) jd[1] = fma(Real(cy(q)) * w, fv(qc), jd[1]);
      if (cz(q)) jd[2] = fma(Real(cz(q)) * w, fv(qc), jd[2]);
    });
  } else {
    Unroll<0, 9>::run([&](auto kc) {
      constexpr int k = decltype(kc)::value, q = pair_first(k), o = opp(q);
      constexpr bool ax = inv_wq(q) == 18;
      const L p = in(std::integral_constant<int, q>{}), m = in(std::integral_constant<int, o>{});
      sd[k] = L::add(p, m);
      sd[9 + k] = L::sub(p, m);
      if constexpr (ax)
        axis = q == 5 ? sd[k] : L::add(axis, sd[k]);
      else
        tot = q == 1 ? sd[k] : L::add(tot, sd[k]);
      const Real dif = sd[9 + k].lo();
      auto take = [&](int i, int c, bool start) {
        if (ax)
          ja[i] = dif;
        else
          jd[i] = start ? dif : (c > 0 ? add_rn(jd[i], dif) : sub_rn(jd[i], dif));
      };
      if (cx(q)) take(0, cx(q), q == 1);
      if (cy(q)) take(1, cy(q), q == 1);
      if (cz(q)) take(2, cz(q), q == 7);
    });
    sd[18] = in(std::integral_constant<int, 0>{});
    tot = L::add(L::add(tot, axis), sd[18]);
  }
  drho = tot.lo();
  sC = tot.hi();
  const Real ir = rcp_as<S>(add_rn(Real(1), drho));
#pragma unroll
  for (int i = 0; i < 3; ++i) V[i] = mul_rn(S::kShift ? jd[i] : add_rn(ja[i], jd[i]), ir);
}

template <class Real>
struct Lat1 {
  __device__ __forceinline__ static Real add(Real a, Real b) { return add_rn(a, b); }
  __device__ __forceinline__ static Real sub(Real a, Real b) { return sub_rn(a, b); }
};

// sum_i c_qi a_i for the axes of direction q, by additions
template <int q, class A, class F>
__device__ __forceinline__ A along(const A (&a)[3], F) {
  constexpr int c[3] = {cx(q), cy(q), cz(q)};
  constexpr int i = c[0] ? 0 : (c[1] ? 1 : 2);                      // first axis
  constexpr int k = (c[0] && c[1]) ? 1 : ((c[2] && i != 2) ? 2 : -1);  // second, or none
  if constexpr (k < 0) {
    static_assert(c[i] == 1, "pair_first lists the positive axis directions");
    return a[i];
  } else if constexpr (c[i] == 1 && c[k] == 1) {
    return F::add(a[i], a[k]);
  } else if constexpr (c[i] == 1) {
    return F::sub(a[i], a[k]);
  } else {
    static_assert(c[k] == 1, "one of a pair's directions has a positive component");
    return F::sub(a[k], a[i]);
  }
}

// x / fl(1/3) in FP32, correctly rounded: the quotient by multiplication with
// 3, the rounded reciprocal of fl(1/3), and one step of Markstein's correction.
__device__ __forceinline__ float div_third(float x) {
  const float q = x * 3.0f;
  return fmaf(fmaf(-wq<float>(0), q, x), 3.0f, q);
}

// Solute collision of one lattice (Eq. equild, BGK) for itd = 1/tau_D, per
// cell. With e = sC / 36 and H = 3 itd e V*, the sum s and the difference d of a
// pair of opposite diagonals become twice e - (1 - itd) (e - s/2) and (1 - itd)/2 d +
// c_q.H (axes: twice e and c_q.H), and the rest direction gives up what the 18
// others gained, 2 itd sum (e - s/2). Roundings then scale with the distance from
// the equilibrium, and a cell keeps its solute to those of the gains. Formed as
// (1 - itd) s/2 + itd e, every collision lost ~1e-8 of the solute in FP32 (tau_D
// 0.6, 0.75), and C was 3e-7 .. 5e-7 from the 64-bit result after 60 steps; now
// 7e-8 .. 9e-8, and FP64 populations of a random medium 2.7e-16 instead of 5.2e-16.
template <class Real>
struct SoluteRows {
  Real e, H[3];
  __device__ __forceinline__ void fold(Real sC, Real itd, Real v0, Real v1, Real v2) {
    e = mul_rn(wq<Real>(1), sC);
    const Real e3 = mul_rn(Real(3), mul_rn(itd, e));
    H[0] = mul_rn(e3, v0);
    H[1] = mul_rn(e3, v1);
    H[2] = mul_rn(e3, v2);
  }
};

// The per-cell arithmetic after streaming: concentration and viscosity,
// colour gradient, V' and the Darcy force, fluid and solute collision,
// stores and exported fields. drho, V are the fluid moments, sC the solute
// total of the arriving h, sd their sums and differences (16-bit storage: fv(q)
// and hv(q) give (f_q - w_q)/w_q and h_q/w_q), kv(r) the rows of K^-1.
//
// Fluid collision (Eqs. equilc1, equilc2, coeffforce1), folded per cell: f~_q -
// w_q = (1 - 1/tau)(f_q - w_q) + w_q b_q with
//   b_q = K + c.W + (c.V')(c.X),   P = rho (1 - 1/(2 tau)),
//   W = 3 (rho/tau V' + P F_e),  Y = 3 (rho/(2 tau) V' + P F_e),  X = 3/eps Y,
//   K = (rho - 1)/tau - V'.Y / eps
// (surface tension: + A eps ((c.F)^2/|F| - |F|), + A eps |F| at rest). Opposite
// directions are formed from the sum s and the difference d of their old
// values as E + O and E - O, E = (1 - 1/tau)/2 s + w (K + (c.V')(c.X)), O = (1 -
// 1/tau)/2 d + w c.W: for a pair of diagonals of both lattices two packed
// additions give the dot products, one fma and two packed fmas E and O, two more
// instructions the solute's part of E (SoluteRows), two packed additions the new
// values: 9 instructions where the unfolded form took ~26. Where the density is away from 1 (E much larger than O: a wood sample
// under pressure) the rounding of E drops out of the momentum: after 60 steps
// at 256x192x64 FP32 u is 4.1e-6 from the 64-bit result, 1.0e-5 before. Without
// the solute the flow is driven by a force at density 1 (O the larger part),
// and the new values are (1 - 1/tau)(f_q - w_q) + w b_q, which keeps the two
// roundings of opposite directions independent. The weights 1/36
// (diagonal), 2/36 (axis) and 12/36 (rest) are folded into the coefficients.
// Every operation is an explicit fma, product or sum, so all kernels that
// inline this round alike.
//
// 16-bit storage keeps the order of operations of FluidCollide (its results
// are compared bit by bit), both lattices in packed instructions.
// VOUT: the cell's bare V and V' are returned in vout[0..2], vout[3..5]
// (for the further solute species of the same thread).
template <class S, int KMODE, bool SOLUTE, bool TENS, bool VOUT = false, class FV, class HV, class KV>
__device__ __forceinline__ void collide_tail(const StepArgs<typename S::Real> &a, unsigned n,
                                             const CellGeo &g, FV fv, HV hv, KV kv,
                                             const Lat<typename S::Real, SOLUTE> (&sd)[Q],
                                             typename S::Real drho,
                                             const typename S::Real (&V)[3], typename S::Real ie,
                                             typename S::Real eps, typename S::Real sC,
                                             typename S::Real gx, typename S::Real gy,
                                             typename S::Real gz,
                                             typename S::Real *vout = nullptr) {
  using Real = typename S::Real;
  using T = typename S::T;
  using L = Lat<Real, SOLUTE>;
  using D = Lat<Real, true>;
  const unsigned N = a.N;
  const Real rho = Real(1) + drho;
  const Real C = SOLUTE ? sC * ie : Real(0);
  Real tau, nu;
  if constexpr (S::kShift) {  // (the order of operations that its results are compared by)
    tau = tau_of(a, C);
    nu = a.visc_law == 0 ? a.nu0 : (tau - Real(0.5)) * Real(1.0 / 3.0);
  } else {
    tau_nu(a, C, tau, nu);
  }
  FluidCollide<Real> fc;
  Real(&Vp)[3] = fc.Vp, (&Fe)[3] = fc.Fe, (&F)[3] = fc.F;
  auto again = [&](int r) { return __ldcg(r < 6 ? a.kinv + size_t(r) * N + n : a.eps + n); };
  velocity_solve_kv<KMODE, S::kShift>(kv, again, eps, nu, V, a.G, a.forch, Vp, Fe);
  Real Fn = Real(0);
  bool st = false;
  F[0] = F[1] = F[2] = Real(0);
  if constexpr (TENS) {
    colour_gradient(a.rhohat, n, g, a.f_wall, a.wall_rho, F);
    Fn = sqrt(F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
    st = Fn > st_threshold<Real>();
  }
  const Real itd = a.inv_tau_D, vs[3] = {Vp[0] + gx, Vp[1] + gy, Vp[2] + gz};
  T *__restrict__ fo = static_cast<T *>(a.f_out) + n;
  if constexpr (S::kShift) {
    fc.drho = drho;
    fc.rho = rho;
    fc.ie = ie;
    fc.uu = Vp[0] * Vp[0] + Vp[1] * Vp[1] + Vp[2] * Vp[2];
    fc.uF = Vp[0] * Fe[0] + Vp[1] * Fe[1] + Vp[2] * Fe[2];
    fc.itau = rcp(tau);
    fc.omt = Real(1) - fc.itau;
    fc.pre = rho * (Real(1) - Real(0.5) * fc.itau);
    fc.st = st;
    fc.Fn = Fn;
    fc.stc = st ? a.A * eps * tau : Real(0);
    fc.iFn = st ? Real(1) / Fn : Real(0);
    const Real sc = Real(S::kScale);
    if constexpr (SOLUTE) {
      // paired layout: the references are drho and sC rounded to FP16, the
      // remainders are formed against the rounded values.
      // f: (f~_q - w_q)/w_q = omt e_q + b_q, stored scale ((f~_q - w_q)/w_q - Rf).
      // h: h~_q/w_q = (1 - 1/tau_D) h_q/w_q + h^eq_q/(w_q tau_D) with
      // h^eq_q/w_q = sC (1 + 3 c_q.v), stored scale (h~_q/w_q - Rh); the rest
      // direction takes sC - sum_{q>0} h^eq_q, divided by its weight, so the
      // weights' rounding adds no solute.
      using T2 = typename S::T2;
      const __half2 r2 = __floats2half2_rn(drho, sC);
      const float2 R = __half22float2(r2);
      T2 *__restrict__ po = static_cast<T2 *>(a.f_out) + n;
      fc.fold(sc, R.x);
      const Real so = sc * fc.omt, sod = sc * (Real(1) - itd), h0 = sc * (itd * sC - R.y),
                 h3 = Real(3) * sc * itd * sC;
      const L om = L::mk(so, sod), up = L::mk(Real(1), h3), down = L::mk(Real(-1), -h3);
      const L uv[3] = {L::mk(Vp[0], vs[0]), L::mk(Vp[1], vs[1]), L::mk(Vp[2], vs[2])};
      Real hsum = Real(0);
      Unroll<0, 9>::run([&](auto kc) {
        constexpr int q = pair_first(decltype(kc)::value), o = opp(q);
        const auto qq = std::integral_constant<int, q>{};
        const auto oo = std::integral_constant<int, o>{};
        const L c = along<q>(uv, L{});
        hsum = fma(Real(2) * wq<Real>(q), sC, hsum);
        Real ev, od;
        fc.template even_odd<q>(c.lo(), ev, od);
        const L e = L::mk(ev, h0), odd = L::mk(od, c.hi());
        const L vq = L::fma(om, L::mk(fv(qq), hv(qq)), L::fma(up, odd, e));
        const L vo = L::fma(om, L::mk(fv(oo), hv(oo)), L::fma(down, odd, e));
        S::st2(po + int(q * N), vq.lo(), vq.hi());
        S::st2(po + int(o * N), vo.lo(), vo.hi());
      });
      const Real he0 = div_third(sC - hsum);
      const auto q0 = std::integral_constant<int, 0>{};
      S::st2(po, fma(so, fv(q0), fc.template br<0>()), fma(sod, hv(q0), sc * (itd * he0 - R.y)));
      reinterpret_cast<__half2 *>(a.rf_out)[n] = r2;
    } else {
      // per unit weight, (f~_q - w_q)/w_q = omt e_q + b_q; stored as the
      // remainder scale ((f~_q - w_q)/w_q - drho)
      fc.fold(sc, drho);
      const Real so = sc * fc.omt;
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        S::template st_raw<q>(fo + int(q * N), fma(so, fv(qc), fc.template br<q>()));
      });
      a.rf_out[n] = float(drho);
    }
  } else {
    constexpr Real w = wq<Real>(1);
    const Real itau = a.visc_law == 0 ? a.itau : rcp1(tau), omt = Real(1) - itau;
    // (FP64 multiplies by rho last, so the factors of a constant tau are uniform;
    // in FP32 their rounding, the same in every cell, doubled the error of u)
    const Real it = w * itau, pf = fma(Real(-0.5), itau, Real(1));
    constexpr bool last = sizeof(Real) == 8;
    const Real r3 = last ? (Real(3) * it) * rho : Real(3) * (it * rho), r15 = Real(0.5) * r3;
    const Real p3 = last ? (Real(3) * w * pf) * rho : Real(3) * w * (rho * pf);
    const Real ie3 = Real(3) * ie;
    Real K, Wv[3], X[3], VY = Real(0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const Real t = mul_rn(p3, Fe[i]), Y = fma(r15, Vp[i], t);
      Wv[i] = fma(r3, Vp[i], t);
      X[i] = mul_rn(ie3, Y);
      VY = fma(Vp[i], Y, VY);
    }
    K = fma(it, drho, -mul_rn(ie, VY));
    Real K0 = K, S2 = Real(0);
    if (TENS && st) {
      const Real ae = w * a.A * eps, ks = ae * Fn;
      K0 = K + ks;
      K -= ks;
      S2 = ae / Fn;
    }
    SoluteRows<Real> so{};
    T *__restrict__ ho = nullptr;
    if constexpr (SOLUTE) {
      so.fold(sC, itd, vs[0], vs[1], vs[2]);
      ho = static_cast<T *>(a.h_out) + n;
    }
    const Real omd = Real(1) - itd;
    Real gained = Real(0);  // by the moving solute, over 2 itd
    const L om = L::mk(omt, omd), half = L::mk(Real(0.5) * omt, Real(0.5) * omd);
    const L W2[3] = {L::mk(Wv[0], so.H[0]), L::mk(Wv[1], so.H[1]), L::mk(Wv[2], so.H[2])};
    const D VX[3] = {D::mk(Vp[0], X[0]), D::mk(Vp[1], X[1]), D::mk(Vp[2], X[2])};
    auto store = [&](auto qc, L v) {
      constexpr int q = decltype(qc)::value;
      S::template st_f<q>(fo + int(q * N), v.lo());
      if constexpr (SOLUTE) S::template st_h<q>(ho + int(q * N), v.hi());
    };
    Unroll<0, 9>::run([&](auto kc) {
      constexpr int k = decltype(kc)::value, q = pair_first(k), o = opp(q);
      L od = along<q>(W2, L{});
      const D vx = along<q>(VX, D{});
      Real ev = fma(vx.lo(), vx.hi(), K);
      if constexpr (TENS) {
        const Real cs = dot_c<q>(F[0], F[1], F[2]);
        ev = fma(S2 * cs, cs, ev);
      }
      L e = L::mk(ev, so.e);  // solute: the equilibrium itself
      if constexpr (inv_wq(q) == 18) {  // weight 2/36
        od = L::add(od, od);
        e = L::add(e, e);
      }
      const auto qq = std::integral_constant<int, q>{};
      const auto oo = std::integral_constant<int, o>{};
      if constexpr (SOLUTE) {
        Real gap;
        e = L::relax(sd[k], e, half.lo(), omd, gap);
        gained = k == 0 ? gap : add_rn(gained, gap);
        od = L::fma(half, sd[9 + k], od);
        store(qq, L::add(e, od));
        store(oo, L::sub(e, od));
      } else {
        store(qq, L::fma(om, L::mk(fv(qq), Real(0)), L::add(e, od)));
        store(oo, L::fma(om, L::mk(fv(oo), Real(0)), L::sub(e, od)));
      }
    });
    const L r0 = sd[18];
    store(std::integral_constant<int, 0>{},
          L::fma(L::mk(omt, Real(-2) * itd), L::mk(r0.lo(), gained),
                 L::mk(mul_rn(Real(12), K0), r0.hi())));
  }
  if (a.fields) write_fields(a.fields, N, n, rho, Vp, C, nu);
  if constexpr (VOUT) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      vout[i] = V[i];
      vout[3 + i] = Vp[i];
    }
  }
}

// The rows of a cell's K^-1, loaded with its other static fields before the
// moments, so that their latency hides behind the gather (inside the velocity
// solve they are a second wait per cell: 256^3 FP32 with a full tensor 0.955 ->
// 0.862 ms, and since the collision needs fewer registers also the diagonal
// tensor, 128^3 FP32 0.1091 -> 0.1084 ms).
template <class Real, int KMODE>
struct KinvRows {
  static constexpr int kRows = KMODE == KM_NONE ? 0 : (KMODE == KM_SPD ? 6 : 3);
  Real v[kRows ? kRows : 1];
  __device__ __forceinline__ void load(const Real *kinv, unsigned N, unsigned n) {
    for (int r = 0; r < kRows; ++r) v[r] = __ldg(kinv + size_t(r) * N + n);
  }
};

// The directions whose pull leaves through one of the given faces.
__host__ __device__ constexpr uint32_t dirs_through(unsigned faces) {
  uint32_t m = 0;
  for (int q = 1; q < Q; ++q)
    if (faces_crossed(q) & faces) m |= 1u << q;
  return m;
}
// The directions that bounce back in a cell, as a mask: sources that are
// solid (link) or behind a wall face.
__device__ __forceinline__ uint32_t bounce_mask(uint32_t link, unsigned walls_on) {
  uint32_t m = link & 0x7ffffu;
#pragma unroll
  for (int f = 0; f < 6; ++f)
    if ((walls_on >> f) & 1u) m |= dirs_through(1u << f);
  return m;
}

// The rules of pressure and velocity faces for the directions of fprs and
// fvel, whose d[q] holds the cell's own f~_qbar: a population entering through a
// pressure face is -f~_qbar + 2 w_q rho_b (1 + 4.5 (c_q.u)^2/eps - 1.5 u.u/eps)
// with rho_b = 3 eps P_face and u the velocity of the cell's own post-collision
// populations; through a velocity face f~_qbar + 6 w_q rho (c_q . u_face), rho
// their density. 16-bit storage: d per unit weight. Out of line: face cells
// are few, and the hot path keeps its registers.
template <class Real>
struct Pops {
  Real v[Q];
};

template <class S>
__device__ __noinline__ Pops<typename S::Real> open_face_rules(
    const StepArgs<typename S::Real> &a, const CellGeo &g, unsigned n, typename S::Real eps,
    uint32_t fvel, uint32_t fprs, Pops<typename S::Real> d) {
  using Real = typename S::Real;
  using T = typename S::T;
  const unsigned N = a.N;
  Real r = Real(0), u0, u1, u2, ie;
  if constexpr (S::kShift) {
    Real j0 = Real(0), j1 = Real(0), j2 = Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      Real v;  // the own f~_q - w_q
      if (a.paired)
        v = wq<Real>(q) * (S::ld2(static_cast<const typename S::T2 *>(a.f_in) + size_t(q) * N + n).x +
                           ld_ref2(a.rf_in + n).x);
      else
        v = S::template ld_f<q>(static_cast<const T *>(a.f_in) + size_t(q) * N + n) +
            wq<Real>(q) * __ldg(a.rf_in + n);
      r += v;
      if (cx(q)) j0 += Real(cx(q)) * v;
      if (cy(q)) j1 += Real(cy(q)) * v;
      if (cz(q)) j2 += Real(cz(q)) * v;
    });
    const Real irho = rcp(Real(1) + r);
    u0 = j0 * irho;
    u1 = j1 * irho;
    u2 = j2 * irho;
    ie = rcp(eps);
  } else {
    Real u[3], s_;
    Lat<Real, false> sd_[Q];
    moments<S, false>(
        [&](auto qc) {
          constexpr int q = decltype(qc)::value;
          return S::template ld_f<q>(static_cast<const T *>(a.f_in) + size_t(q) * N + n);
        },
        [&](auto) { return Real(0); }, r, s_, u, sd_);
    u0 = u[0];
    u1 = u[1];
    u2 = u[2];
    ie = rcp1(eps);
  }
  const Real rho = Real(1) + r;
  const Real uu = u0 * u0 + u1 * u1 + u2 * u2;
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const Real own = S::kShift ? d.v[q] * wq<Real>(q) : d.v[q];
    Real v = own;
    if ((fprs >> q) & 1u) {
      // rho_b - 1 from 3P = hi + lo with one rounding of eps hi - 1
      const int fi = crossed_face<q>(g, a.f_press);
      const Real rbm1 = fma(eps, __ldg(a.face + fi), Real(-1)) + eps * __ldg(a.face + 24 + fi);
      const Real rb = Real(1) + rbm1;
      const Real cu = dot_c<q>(u0, u1, u2);
      const Real e = wq<Real>(q) * (rbm1 + rb * (Real(4.5) * ie * cu * cu - Real(1.5) * ie * uu));
      v = Real(2) * e - own;
    } else if ((fvel >> q) & 1u) {
      const Real *uf = a.face + 6 + 3 * crossed_face<q>(g, a.f_vel);
      const Real cub = dot_c<q>(__ldg(uf), __ldg(uf + 1), __ldg(uf + 2));
      v = own + Real(6) * wq<Real>(q) * rho * cub;
    }
    d.v[q] = S::kShift ? v * Real(inv_wq(q)) : v;
  });
  return d;
}

// One step of a cell from global memory: stream f (and h), moments,
// viscosity, colour gradient, V' and the Darcy force, fluid and solute
// collision, store; accumulates the cell's flux and totals. 16-bit storage
// with solute (the paired layout): one 32-bit load brings f_q and h_q of a
// source cell, one more its reference pair, and both lattices are gathered
// per unit weight, d[q] = (f_q - w_q)/w_q and hh[q] = h_q/w_q (remainder + the
// source's reference).
template <class S, int KMODE, bool SOLUTE, int FEAT = 0>
__device__ __forceinline__ void update_cell(const StepArgs<typename S::Real> &a, unsigned x,
                                            unsigned y, unsigned z, unsigned n, uint32_t link,
                                            typename S::Real &fin_acc,
                                            typename S::Real &fout_acc, typename S::Real &drho,
                                            typename S::Real &sC, bool &open_face,
                                            typename S::Real *vout = nullptr) {
  using Real = typename S::Real;
  using T = typename S::T;
  constexpr bool kPair = S::kShift && SOLUTE;
  const unsigned N = a.N;
  const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
  Real d[Q], hh[SOLUTE ? Q : 1];
  // element of row `row` of a population buffer at n + off
  auto at = [&](auto e, const void *base, int row, int off) {
    using E = decltype(e);
    return static_cast<const E *>(base) + n + (row * int(N) + off);
  };
  auto both = [&](auto qc, int row, int off) {
    [[maybe_unused]] constexpr int q = decltype(qc)::value;
    if constexpr (kPair) {
      const float2 p = S::ld2(at(typename S::T2{}, a.f_in, row, off));
      const float2 r = ld_ref2(a.rf_in + n + off);
      const auto v = Lat<Real, true>::add(Lat<Real, true>::mk(p.x, p.y), Lat<Real, true>::mk(r.x, r.y));
      d[q] = v.lo();
      hh[SOLUTE ? q : 0] = v.hi();
    }
  };
  auto ld_f = [&](auto qc, int row, int off) -> Real {  // the row of q or of opp(q): same weight
    [[maybe_unused]] constexpr int q = decltype(qc)::value;
    if constexpr (kPair)
      return S::ld2(at(typename S::T2{}, a.f_in, row, off)).x + ld_ref2(a.rf_in + n + off).x;
    else if constexpr (S::kShift)
      return S::template ld_e<q>(at(T{}, a.f_in, row, off)) + __ldg(a.rf_in + n + off);
    else
      return S::template ld_f<q>(at(T{}, a.f_in, row, off));
  };
  auto ld_h = [&](auto qc, int row, int off) -> Real {
    [[maybe_unused]] constexpr int q = decltype(qc)::value;
    if constexpr (kPair)
      return S::ld2(at(typename S::T2{}, a.f_in, row, off)).y + ld_ref2(a.rf_in + n + off).y;
    else
      return S::template ld_h<q>(at(T{}, a.h_in, row, off));
  };
  Real eps, gx = Real(0), gy = Real(0), gz = Real(0);
  KinvRows<Real, KMODE> kr;
  auto statics = [&]() {
    eps = __ldg(a.eps + n);
    if constexpr (SOLUTE) {
      gx = __ldg(a.geps + n);
      gy = __ldg(a.geps + N + n);
      gz = __ldg(a.geps + 2 * size_t(N) + n);
    }
    kr.load(a.kinv, N, n);
  };
  const unsigned s_open = a.s_inlet | a.s_outlet;
  open_face = SOLUTE && (g.onface & s_open) != 0;
  const unsigned open = ((FEAT & FEAT_OPEN) ? a.f_press | a.f_vel : 0u) | (SOLUTE ? s_open : 0u);
  const unsigned walls = a.f_wall | (SOLUTE ? a.s_wall : 0u);
  if (!(g.onface & open)) {
    // Every lane first loads from the cells at n - c_q, whatever is there (the
    // wrapped source is always a cell of the lattice): a warp keeps its 38
    // population rows in flight together, and the link word travels with
    // them. The directions that bounce back are loaded again afterwards. (When
    // the link word decided the addresses, a warp of a medium with 10 % solid
    // cells waited for it, then for a gather of its plain lanes, then for one
    // of its lanes beside solid cells.)
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if constexpr (kPair)
        both(qc, q, src_delta<q>(g));
      else
        d[q] = ld_f(qc, q, src_delta<q>(g));
    });
    if constexpr (SOLUTE && !kPair)
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        hh[q] = ld_h(qc, q, src_delta<q>(g));
      });
    statics();
    if (link != 0 || (g.onface & walls)) {
      const uint32_t mf = bounce_mask(link, g.onface & a.f_wall);
      const uint32_t mh = SOLUTE ? bounce_mask(link, g.onface & a.s_wall) : mf;
      Unroll<1, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if (kPair && ((mf & mh) >> q & 1u)) {
          both(qc, opp(q), 0);
        } else {
          if ((mf >> q) & 1u) d[q] = ld_f(qc, opp(q), 0);
          if (SOLUTE && ((mh >> q) & 1u)) hh[SOLUTE ? q : 0] = ld_h(qc, opp(q), 0);
        }
      });
    }
  } else {
    // On inlet, outlet, pressure or velocity faces: the class of every
    // direction as masks (walls take precedence, then velocity, then pressure;
    // for the solute inlets, then outlets), so that all loads go out together
    // without a branch per direction. In a small lattice these few warps are
    // the longest chain of a step.
    statics();
    const uint32_t solid = link & 0x7ffffu;
    const uint32_t fw = bounce_mask(0u, g.onface & a.f_wall);
    uint32_t fvel = 0, fprs = 0;
    if constexpr ((FEAT & FEAT_OPEN) != 0) {
      fvel = bounce_mask(0u, g.onface & a.f_vel) & ~fw;
      fprs = bounce_mask(0u, g.onface & a.f_press) & ~(fw | fvel);
    }
    // the own population of the opposite direction: bounce-back, and what the
    // pressure and velocity rules start from
    const uint32_t fown = fw | fvel | fprs | solid;
    const uint32_t hw = SOLUTE ? bounce_mask(0u, g.onface & a.s_wall) : 0u;
    const uint32_t hin = SOLUTE ? bounce_mask(0u, g.onface & a.s_inlet) & ~hw : 0u;
    const uint32_t hout = SOLUTE ? bounce_mask(0u, g.onface & a.s_outlet) & ~(hw | hin) : 0u;
    const uint32_t hown = hw | hin | (solid & ~hout);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const bool b = (fown >> q) & 1u;
      d[q] = ld_f(qc, b ? opp(q) : q, b ? 0 : src_delta<q>(g));
    });
    if constexpr (SOLUTE)
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const bool b = (hown >> q) & 1u;
        hh[q] = ld_h(qc, b ? opp(q) : q, (b || ((hout >> q) & 1u)) ? 0 : src_delta<q>(g));
      });
    if constexpr ((FEAT & FEAT_OPEN) != 0) {
      if (g.onface & (a.f_press | a.f_vel)) {
        Pops<Real> o;
        Unroll<0, Q>::run([&](auto qc) { o.v[decltype(qc)::value] = d[decltype(qc)::value]; });
        o = open_face_rules<S>(a, g, n, eps, fvel, fprs, o);
        Unroll<0, Q>::run([&](auto qc) { d[decltype(qc)::value] = o.v[decltype(qc)::value]; });
      }
    }
    if constexpr (SOLUTE) {
      // 16-bit paired values are per unit weight, their fluxes carry the weights
      Real V[3], r_, s_;
      Lat<Real, false> sd_[Q];
      moments<S, false>([&](auto qc) { return d[decltype(qc)::value]; },
                        [&](auto) { return Real(0); }, r_, s_, V, sd_);
      const Real vi0 = V[0] + gx, vi1 = V[1] + gy, vi2 = V[2] + gz;
      const bool counts = !(link >> 31);
      Unroll<1, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        constexpr Real wu = kPair ? Real(1) : wq<Real>(q), wf = kPair ? wq<Real>(q) : Real(1);
        if ((hin >> q) & 1u) {
          // entering through an inlet face: h^eq at C_in with the cell's bare
          // streamed velocity plus D grad(eps)/eps
          const Real cv = dot_c<q>(vi0, vi1, vi2);
          const Real v = wu * eps * a.C_in * (Real(1) + Real(3) * cv);
          const Real f = wf * (v - hh[q]);
          if (counts) fin_acc += f;
          hh[q] = v;
        } else if ((hout >> q) & 1u) {
          // outlet: the cell's own post-collision value (zero gradient)
          const Real f = wf * (ld_h(qc, opp(q), 0) - hh[q]);
          if (counts) fout_acc += f;
        }
      });
    }
  }
  if (link >> 31) return;  // impermeable: never updated
  Real V[3];
  auto fv = [&](auto qc) { return d[decltype(qc)::value]; };
  auto hv = [&](auto qc) { return hh[SOLUTE ? decltype(qc)::value : 0]; };
  Lat<Real, SOLUTE> sd[Q];
  moments<S, SOLUTE>(fv, hv, drho, sC, V, sd);
  const Real ie = rcp_as<S>(eps);
  collide_tail<S, KMODE, SOLUTE, (FEAT & FEAT_TENS) != 0, (FEAT & FEAT_SPEC) != 0>(
      a, n, g, fv, hv, [&](int r) { return kr.v[r]; }, sd, drho, V, ie, eps, sC, gx, gy, gz, vout);
}

// Solute species sp >= 1 of one cell, after the fluid and species 0 of the
// same step (Eqs. equild, boltzeqD for each species, reading R24): each
// species is its own D3Q19 lattice with its own tau_D and inlet
// concentration; all share the cell's V' (vel[3..5]) and, for populations
// entering through an inlet face, its bare streamed velocity V (vel[0..2]).
// The gather with its boundary classes, C = sum_q h_q / eps, h^eq at V* = V' +
// D_s grad(eps)/eps with the rest component as the remainder, BGK.
template <class S>
__device__ __forceinline__ void species_update(const StepArgs<typename S::Real> &a, int sp,
                                               unsigned x, unsigned y, unsigned z, unsigned n,
                                               uint32_t link, const typename S::Real (&vel)[6],
                                               typename S::Real &fin_acc,
                                               typename S::Real &fout_acc, typename S::Real &sC,
                                               bool &open_face) {
  using Real = typename S::Real;
  using T = typename S::T;
  const unsigned N = a.N;
  const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
  // the paired layout keeps species 0 with f, so the h buffers start at species 1
  const size_t off = size_t(sp - a.paired) * Q * N;
  const T *__restrict__ hb = static_cast<const T *>(a.h_in) + off + n;
  T *__restrict__ ho = static_cast<T *>(a.h_out) + off + n;
  const float *rh_in = S::kShift ? a.rh_in + size_t(sp) * N : nullptr;
  const Real eps = __ldg(a.eps + n);
  const Real ratio = __ldg(a.spec + 16 + sp);  // D_s / D_0 (geps holds D_0 grad(eps)/eps)
  const Real gx = ratio * __ldg(a.geps + n), gy = ratio * __ldg(a.geps + N + n),
             gz = ratio * __ldg(a.geps + 2 * size_t(N) + n);
  const Real C_in = __ldg(a.spec + 8 + sp), itd = __ldg(a.spec + sp);
  const unsigned s_open = a.s_inlet | a.s_outlet;
  open_face = (g.onface & s_open) != 0;
  Real hh[Q];
  if (link == 0 && !(g.onface & (a.s_wall | s_open))) {
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      hh[q] = S::template ld_h<q>(hb + (int(q * N) + src_delta<q>(g)));
      if constexpr (S::kShift) hh[q] += wq<Real>(q) * __ldg(rh_in + (long long)n + src_delta<q>(g));
    });
  } else {
    const Real vi0 = vel[0] + gx, vi1 = vel[1] + gy, vi2 = vel[2] + gz;
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const int cls = solute_class<q>(g, link, a.s_wall, a.s_inlet, a.s_outlet);
      Real v;
      const Real own = S::kShift ? wq<Real>(q) * __ldg(rh_in + n) : Real(0);
      if (cls == PULL_CELL) {
        v = S::template ld_h<q>(hb + (int(q * N) + src_delta<q>(g)));
        if constexpr (S::kShift) v += wq<Real>(q) * __ldg(rh_in + (long long)n + src_delta<q>(g));
      } else if (cls == PULL_BOUNCE) {
        v = S::template ld_h<opp(q)>(hb + int(opp(q) * N)) + own;
      } else if (cls == PULL_INLET) {
        const Real cv = dot_c<q>(vi0, vi1, vi2);
        v = wq<Real>(q) * eps * C_in * (Real(1) + Real(3) * cv);
        fin_acc += v - (S::template ld_h<opp(q)>(hb + int(opp(q) * N)) + own);
      } else {
        v = S::template ld_h<q>(hb + int(q * N)) + own;
        fout_acc += (S::template ld_h<opp(q)>(hb + int(opp(q) * N)) + own) - v;
      }
      hh[q] = v;
    });
  }
  if constexpr (S::kShift) {
    // weighted rows against an FP32 reference: the remainder h~_q - w_q sC
    Unroll<0, Q>::run([&](auto qc) { sC += hh[decltype(qc)::value]; });
    const Real vs0 = vel[3] + gx, vs1 = vel[4] + gy, vs2 = vel[5] + gz;
    Real hsum = Real(0);
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real cv = dot_c<q>(vs0, vs1, vs2);
      const Real heq = wq<Real>(q) * sC * (Real(1) + Real(3) * cv);
      hsum += heq;
      const Real h = hh[q];
      S::template st_h<q>(ho + int(q * N), h + (heq - h) * itd - wq<Real>(q) * sC);
    });
    const Real h = hh[0];
    S::template st_h<0>(ho, h + ((sC - hsum) - h) * itd - wq<Real>(0) * sC);
    a.rh_out[size_t(sp) * N + n] = float(sC);
  } else {
    // the same operations as species 0's (moments, collide_tail), so that
    // equal species stay bit-identical
    Real diag = Real(0), axis = Real(0), dif[9];
    Unroll<0, 9>::run([&](auto kc) {
      constexpr int k = decltype(kc)::value, q = pair_first(k), o = opp(q);
      const Real p = add_rn(hh[q], hh[o]);
      dif[k] = sub_rn(hh[q], hh[o]);
      hh[q] = p;  // the pair's sum
      if (inv_wq(q) == 18)
        axis = q == 5 ? p : add_rn(axis, p);
      else
        diag = q == 1 ? p : add_rn(diag, p);
    });
    sC = add_rn(add_rn(diag, axis), hh[0]);
    SoluteRows<Real> so;
    so.fold(sC, itd, vel[3] + gx, vel[4] + gy, vel[5] + gz);
    const Real om = Real(1) - itd, half = Real(0.5) * om;
    Real gained = Real(0);
    Unroll<0, 9>::run([&](auto kc) {
      constexpr int k = decltype(kc)::value, q = pair_first(k), o = opp(q);
      Real od = along<q>(so.H, Lat1<Real>{}), e = so.e;
      if (inv_wq(q) == 18) {
        od = add_rn(od, od);
        e = add_rn(e, e);
      }
      const Real gap = fma(Real(-0.5), hh[q], e);
      gained = k == 0 ? gap : add_rn(gained, gap);
      e = fma(-om, gap, e);
      od = fma(half, dif[k], od);
      S::template st_h<q>(ho + int(q * N), add_rn(e, od));
      S::template st_h<o>(ho + int(o * N), sub_rn(e, od));
    });
    S::template st_h<0>(ho, fma(Real(-2) * itd, gained, hh[0]));
  }
  if (a.fields) a.fields[(5 + size_t(sp)) * N + n] = float(sC * rcp(eps));
}

// The cell of thread `tid` of block (bx, by, bz) of a per-cell launch with
// rows of `row` threads, and its warp's number in the launch (its flux slot).
// Two mappings. Rows: block (row, STEP_BLOCK/row), grid (ceil(nx/row),
// ceil(ny/(STEP_BLOCK/row)), nz), a warp covers 32 consecutive x of one row
// (nothing to divide). Linear (a.linear): the threads of the launch take the
// cells in the order of n. Where the rows do not fill whole warps the row
// mapping leaves lanes idle (half of them at nx = 16, a warp in four at nx =
// 96), and its rows start inside a 128-byte line; cell_shape picks.
struct CellIndex {
  unsigned x, y, z, n, warp;
  bool in;
};
template <class Real>
__device__ __forceinline__ CellIndex cell_index(const StepArgs<Real> &a, unsigned bx, unsigned by,
                                                unsigned bz, unsigned gx, unsigned gy, unsigned row,
                                                unsigned tx, unsigned ty,
                                                unsigned threads = STEP_BLOCK) {
  CellIndex c;
  if (a.linear) {
    const unsigned tid = ty * row + tx;
    c.n = bx * threads + tid;
    c.in = c.n < a.N;
    const unsigned yz = a.by_nx.div(c.n);
    c.x = c.n - yz * unsigned(a.nx);
    c.z = a.by_ny.div(yz);
    c.y = yz - c.z * unsigned(a.ny);
    c.warp = c.n >> 5;
  } else {
    c.x = bx * row + tx;
    c.y = by * (STEP_BLOCK / row) + ty;
    c.z = bz;
    c.in = c.x < unsigned(a.nx) && c.y < unsigned(a.ny);
    c.n = c.x + unsigned(a.nx) * (c.y + unsigned(a.ny) * c.z);
    c.warp = ((bz * gy + by) * gx + bx) * (STEP_BLOCK / 32) + ((ty * row + tx) >> 5);
  }
  return c;
}

// Resident 128-thread blocks per SM of the per-cell kernel (registers a thread).
// The kernel is bound by loads in flight, so warps are traded against registers
// that keep a cell's ~48 loads together. Measured on GB300, ms per step with 4 /
// 5 / 6 / 7 blocks: 128^3 FP32 diagonal 0.1064 / 0.1050 / 0.1091 / 0.1134,
// Forchheimer 0.1134 / 0.1064 / 0.1144 / 0.1180, 117x83x101 with 10 % solid cells
// 0.0908 / 0.0893 / 0.0963 / 0.1004, 256^3 with a full tensor 0.838 / 0.833 / 0.902
// / 0.909, 256x192x64 with pressure faces 0.1663 / 0.1650 / 0.1731 / 0.1796, three
// species 0.2249 / 0.2118 / 0.2249 / 0.2242 (6 took 0.2201 before); 256^3 FP16 with a
// full tensor 0.725 / 0.666 / 0.616 / 0.616, with a diagonal one 0.678 / 0.573 at 6 /
// 7, BF16 0.754 / 0.740 / 0.640 / 0.702. The batched kernel takes 6 (15 lattices FP32
// 0.269 / 0.286 / 0.245 / 0.256, 24 of 32^3 FP16 0.0509 / 0.0514 / 0.0430 / 0.0445).
// FP64 populations take twice the registers, and its pipe is busy with a few warps.
template <class S, bool SOLUTE, int FEAT>
constexpr int step_blocks() {
  if (sizeof(typename S::Real) == 8) return 3;
  if (std::is_same<S, StoreF16>::value && SOLUTE && FEAT == 0) return 7;
  return S::kShift || !SOLUTE ? 6 : 5;
}
// One time step for every non-solid cell (see update_cell; launch shapes at
// cell_index).
template <class S, int KMODE, bool SOLUTE, int FEAT>
__global__ void __launch_bounds__(STEP_BLOCK, step_blocks<S, SOLUTE, FEAT>()) step_kernel(const StepArgs<typename S::Real> a) {
  using Real = typename S::Real;
  const CellIndex c = cell_index(a, blockIdx.x, blockIdx.y, blockIdx.z, gridDim.x, gridDim.y,
                                 blockDim.x, threadIdx.x, threadIdx.y, blockDim.x);
  const unsigned x = c.x, y = c.y, z = c.z, n = c.n, warp_gid = c.warp;
  const uint32_t link = (c.in && a.link) ? __ldg(a.link + n) : 0u;
  Real fin_acc = Real(0), fout_acc = Real(0), drho = Real(0), sC = Real(0);
  bool open_face = false;
  Real vel[6];
  if (c.in)  // returns early in solid cells
    update_cell<S, KMODE, SOLUTE, FEAT>(a, x, y, z, n, link, fin_acc, fout_acc, drho, sC,
                                        open_face, (FEAT & FEAT_SPEC) ? vel : nullptr);
  [[maybe_unused]] const bool live = c.in && !(link >> 31);
  warp_reductions(a, warp_gid, open_face, fin_acc, fout_acc, drho, sC);
  if constexpr ((FEAT & FEAT_SPEC) != 0) {
    // further species, each with its per-warp flux slots and finite check
    const unsigned lane = threadIdx.x & 31u;
    for (int sp = 1; sp < a.species; ++sp) {
      Real fin_s = Real(0), fout_s = Real(0), sC_s = Real(0);
      bool of = false;
      if (live) species_update<S>(a, sp, x, y, z, n, link, vel, fin_s, fout_s, sC_s, of);
      if (a.flux && __any_sync(0xffffffffu, of)) {
        const Real si = warp_sum(fin_s), so = warp_sum(fout_s);
        if (lane == 0) {
          double *slot = a.flux_slots + size_t(sp) * a.slot_stride + 2 * size_t(warp_gid);
          slot[0] += double(si);
          slot[1] += double(so);
        }
      }
      if (a.reduce) finite_check(a.state, sC_s, Real(0));
    }
  }
}

// Post-stream density for the colour gradient (flowchart: stream -> moments
// -> gradient): rhohat = sum_q f_q(x - c_q), solid cells = wall_rho.
template <class S>
__global__ void __launch_bounds__(BLOCK) rhohat_kernel(const StepArgs<typename S::Real> a,
                                                       typename S::Real *rhohat) {
  using Real = typename S::Real;
  const unsigned n = blockIdx.x * BLOCK + threadIdx.x;
  if (n >= a.N) return;
  uint32_t link = a.link ? __ldg(a.link + n) : 0u;
  if (link >> 31) {
    rhohat[n] = a.wall_rho;
    return;
  }
  const CellGeo g = cell_geo(n, a.nx, a.ny, a.nz);
  Real d[Q];
  gather_f<S>(static_cast<const typename S::T *>(a.f_in), a.N, n, g, link, a.f_wall, d, a.rf_in,
              a.paired != 0);
  Real s = Real(0);
  Unroll<0, Q>::run([&](auto qc) { s += d[decltype(qc)::value]; });
  rhohat[n] = Real(1) + s;
}

// ------------------------------------------------------------------------
// Initialisation (flowchart step c): f = f^eq, h = h^eq. The first step
// writes the other buffer of every updated cell; only the cells that no step
// writes (solid, empty) are set in both.
// ------------------------------------------------------------------------
template <class Real>
struct InitArgs {
  const float *rho0, *u0, *C0, *f_scale;  // device copies of the caller's arrays
  const uint8_t *type;                      // NULL unless free surface
};

template <class S, int KMODE, bool SOLUTE>
__global__ void __launch_bounds__(BLOCK) init_kernel(const StepArgs<typename S::Real> a,
                                                     const InitArgs<typename S::Real> in) {
  using Real = typename S::Real;
  using T = typename S::T;
  const unsigned n = blockIdx.x * BLOCK + threadIdx.x;
  const unsigned N = a.N;
  if (n >= N) return;
  T *fout = static_cast<T *>(a.f_out);
  T *fout2 = static_cast<T *>(const_cast<void *>(a.f_in));
  const bool solid = a.link && (__ldg(a.link + n) >> 31);
  const bool empty = in.type && in.type[n] == CELL_EMPTY;
  if constexpr (S::kShift && SOLUTE) {
    // paired layout: (f, h) remainders per direction, FP16 reference pairs
    using T2 = typename S::T2;
    T2 *p1 = static_cast<T2 *>(a.f_out) + n;
    T2 *p0 = static_cast<T2 *>(const_cast<void *>(a.f_in)) + n;
    if (solid || empty) {
      // absolute populations 0: references (-1, 0), remainders 0
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        S::st2(p1 + size_t(q) * N, 0.0f, 0.0f);
        S::st2(p0 + size_t(q) * N, 0.0f, 0.0f);
      });
      const __half2 r2 = __floats2half2_rn(-1.0f, 0.0f);
      reinterpret_cast<__half2 *>(a.rf_out)[n] = r2;
      reinterpret_cast<__half2 *>(const_cast<float *>(a.rf_in))[n] = r2;
      if (a.fields) zero_fields(a.fields, N, n);
      return;
    }
  }
  if (solid || empty) {
    // absolute populations 0 (FP16/BF16: reference -1, remainders 0)
    const Real shift = S::kShift ? Real(-1) : Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      S::template st_f<q>(fout + size_t(q) * N + n, -wq<Real>(q) - wq<Real>(q) * shift);
      S::template st_f<q>(fout2 + size_t(q) * N + n, -wq<Real>(q) - wq<Real>(q) * shift);
    });
    if constexpr (S::kShift) {
      a.rf_out[n] = -1.0f;
      const_cast<float *>(a.rf_in)[n] = -1.0f;
      if (SOLUTE) {
        a.rh_out[n] = 0.0f;
        const_cast<float *>(a.rh_in)[n] = 0.0f;
      }
    }
    if (SOLUTE) {
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        S::template st_h<q>(static_cast<T *>(a.h_out) + size_t(q) * N + n, Real(0));
        S::template st_h<q>(const_cast<T *>(static_cast<const T *>(a.h_in)) + size_t(q) * N + n,
                            Real(0));
      });
    }
    if (a.fields) zero_fields(a.fields, N, n);
    return;
  }
  const CellGeo g = cell_geo(n, a.nx, a.ny, a.nz);
  const Real rho = Real(in.rho0[n]);
  const Real u[3] = {Real(in.u0[3 * size_t(n)]), Real(in.u0[3 * size_t(n) + 1]),
                     Real(in.u0[3 * size_t(n) + 2])};
  const Real eps = a.eps[n];
  const Real C = SOLUTE ? Real(in.C0[n]) : Real(0);
  const Real tau = tau_of(a, C);  // a.t = 0
  FluidCollide<Real> fc;
  fc.F[0] = fc.F[1] = fc.F[2] = Real(0);
  if (a.A != Real(0)) colour_gradient(a.rhohat, n, g, a.f_wall, a.wall_rho, fc.F);
  fc.drho = rho - Real(1);
  fc.rho = rho;
  fc.ie = Real(1) / eps;
  fc.Vp[0] = u[0]; fc.Vp[1] = u[1]; fc.Vp[2] = u[2];
  fc.uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  fc.Fn = sqrt(fc.F[0] * fc.F[0] + fc.F[1] * fc.F[1] + fc.F[2] * fc.F[2]);
  fc.st = (a.A != Real(0)) && fc.Fn > st_threshold<Real>();
  fc.stc = fc.st ? a.A * eps * tau : Real(0);
  fc.iFn = fc.st ? Real(1) / fc.Fn : Real(0);
  Real devs[Q];
  Real dsum = Real(0);
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    Real dev = fc.template feq_dev<q>();
    if (in.f_scale) {
      const Real sc = Real(in.f_scale[size_t(q) * N + n]);
      dev = (dev + wq<Real>(q)) * sc - wq<Real>(q);
    }
    devs[q] = dev;
    dsum += dev;
  });
  if constexpr (S::kShift && SOLUTE) {
    const Real vs0 = u[0] + a.geps[n], vs1 = u[1] + a.geps[N + n], vs2 = u[2] + a.geps[2 * size_t(N) + n];
    Real hs[Q];
    Real hsum = Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real cv = dot_c<q>(vs0, vs1, vs2);
      hs[q] = wq<Real>(q) * eps * C * (Real(1) + Real(3) * cv);
      hsum += hs[q];
    });
    // remainders per unit weight against the FP16-rounded references
    const __half2 r2 = __floats2half2_rn(dsum, hsum);
    const float2 R = __half22float2(r2);
    using T2 = typename S::T2;
    T2 *p0 = static_cast<T2 *>(const_cast<void *>(a.f_in)) + n;
    const Real sc = Real(S::kScale);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real gf = sc * (devs[q] * Real(inv_wq(q)) - R.x);
      const Real gh = sc * (hs[q] * Real(inv_wq(q)) - R.y);
      S::st2(p0 + size_t(q) * N, gf, gh);
    });
    reinterpret_cast<__half2 *>(const_cast<float *>(a.rf_in))[n] = r2;
    if (a.fields) write_fields(a.fields, N, n, rho, u, C, (tau - Real(0.5)) / Real(3));
    return;
  }
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const Real v = devs[q] - (S::kShift ? wq<Real>(q) * dsum : Real(0));
    S::template st_f<q>(fout2 + size_t(q) * N + n, v);
  });
  if constexpr (S::kShift) const_cast<float *>(a.rf_in)[n] = float(dsum);
  if (SOLUTE) {
    const Real vs0 = u[0] + a.geps[n], vs1 = u[1] + a.geps[N + n], vs2 = u[2] + a.geps[2 * size_t(N) + n];
    Real hs[Q];
    Real hsum = Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real cv = dot_c<q>(vs0, vs1, vs2);
      hs[q] = wq<Real>(q) * eps * C * (Real(1) + Real(3) * cv);
      hsum += hs[q];
    });
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real h = hs[q] - (S::kShift ? wq<Real>(q) * hsum : Real(0));
      S::template st_h<q>(const_cast<T *>(static_cast<const T *>(a.h_in)) + size_t(q) * N + n, h);
    });
    if constexpr (S::kShift) const_cast<float *>(a.rh_in)[n] = float(hsum);
  }
  if (a.fields) write_fields(a.fields, N, n, rho, u, C, (tau - Real(0.5)) / Real(3));
}

// ------------------------------------------------------------------------
// Populations <-> absolute FP64, totals and the neighbour export.
// ------------------------------------------------------------------------
// The reference of cell n in a view (0 without references).
__device__ __forceinline__ double pop_ref(const PopView &v, unsigned n) {
  if (!v.ref) return 0.0;
  if (v.ref_pair) {
    const __half2 r = static_cast<const __half2 *>(v.ref)[n];
    return double(v.off ? __high2float(r) : __low2float(r));
  }
  return double(static_cast<const float *>(v.ref)[n]);
}
template <class S>
__device__ __forceinline__ typename S::T pop_at(const PopView &v, size_t i) {
  return static_cast<const typename S::T *>(v.p)[size_t(v.stride) * i + v.off];
}

template <class S>
__global__ void to_f64_kernel(const PopView v, double *dst, unsigned N, int lattice) {
  const size_t i = size_t(blockIdx.x) * BLOCK + threadIdx.x;
  if (i >= size_t(Q) * N) return;
  const int q = int(i / N);
  const double r = pop_ref(v, unsigned(i % N));
  dst[i] = lattice == 0 ? S::to_f(pop_at<S>(v, i), q, r) : S::to_h(pop_at<S>(v, i), q, r);
}

// per cell: the reference of given FP64 populations (sum of f_q - w_q, or of
// h_q), stored rounded to the view's reference type
static __global__ void ref_from_f64_kernel(const double *src, unsigned N, int lattice,
                                           const PopView v) {
  const unsigned n = blockIdx.x * BLOCK + threadIdx.x;
  if (n >= N) return;
  double s = 0.0;
  for (int q = 0; q < Q; ++q) s += src[size_t(q) * N + n] - (lattice == 0 ? wq<double>(q) : 0.0);
  if (v.ref_pair)
    static_cast<__half *>(const_cast<void *>(v.ref))[2 * size_t(n) + v.off] = __float2half_rn(float(s));
  else
    static_cast<float *>(const_cast<void *>(v.ref))[n] = float(s);
}

template <class S>
__global__ void from_f64_kernel(const double *src, const PopView v, unsigned N, int lattice) {
  const size_t i = size_t(blockIdx.x) * BLOCK + threadIdx.x;
  if (i >= size_t(Q) * N) return;
  const int q = int(i / N);
  const double r = pop_ref(v, unsigned(i % N));
  static_cast<typename S::T *>(const_cast<void *>(v.p))[size_t(v.stride) * i + v.off] =
      lattice == 0 ? S::from_f(src[i], q, r) : S::from_h(src[i], q, r);
}

// Per-block FP64 sums of the fluid mass and the solute over non-solid cells,
// each block taking cells blockIdx.x*BLOCK + tid + k*gridDim.x*BLOCK. A
// cell's 19 stored values are summed in the collision type as deviations
// (FP32 / FP64 storage: f_q - w_q, h_q; 16-bit: the remainders times w_q),
// then mass = 1 + reference + sum, solute = reference + sum in FP64; the
// cell sums, the block's shuffle tree and the finish are FP64.
template <class S>
__global__ void __launch_bounds__(BLOCK) totals_kernel(const PopView f, const PopView h,
                                                       const uint32_t *link, unsigned N,
                                                       double *partials) {
  using Real = typename S::Real;
  __shared__ double sh[BLOCK / 32][2];
  double m = 0.0, s = 0.0;
  for (unsigned n = blockIdx.x * BLOCK + threadIdx.x; n < N; n += gridDim.x * BLOCK) {
    if (link && (link[n] >> 31)) continue;
    if constexpr (S::kShift)
      if (f.ref_pair && h.p == f.p) {
        // the paired layout: f and species 0 in one load (half of each 4-byte
        // pair was loaded twice, 139 us at 160^3 FP16)
        using T2 = typename S::T2;
        Real a = Real(0), b = Real(0);
        Unroll<0, Q>::run([&](auto qc) {
          constexpr int q = decltype(qc)::value;
          const T2 p = static_cast<const T2 *>(f.p)[size_t(q) * N + n];
          a += S::template cv_f<q>(p.x);
          b += S::template cv_h<q>(p.y);
        });
        m += 1.0 + pop_ref(f, n) + double(a);
        s += pop_ref(h, n) + double(b);
        continue;
      }
    Real a = Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      a += S::template cv_f<q>(pop_at<S>(f, size_t(q) * N + n));
    });
    m += 1.0 + pop_ref(f, n) + double(a);
    if (h.p) {
      Real b = Real(0);
      Unroll<0, Q>::run([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        b += S::template cv_h<q>(pop_at<S>(h, size_t(q) * N + n));
      });
      s += pop_ref(h, n) + double(b);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    m += __shfl_down_sync(0xffffffffu, m, o);
    s += __shfl_down_sync(0xffffffffu, s, o);
  }
  const unsigned w = threadIdx.x >> 5;
  if ((threadIdx.x & 31u) == 0) {
    sh[w][0] = m;
    sh[w][1] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tm = 0.0, ts = 0.0;
    for (unsigned k = 0; k < BLOCK / 32; ++k) {
      tm += sh[k][0];
      ts += sh[k][1];
    }
    partials[2 * size_t(blockIdx.x)] = tm;
    partials[2 * size_t(blockIdx.x) + 1] = ts;
  }
}

// Fixed-order sum of nblk x K partials by blocks of FINISH_THREADS threads
// into a set of K sums per block (thread t of the launch sums partials t, t +
// threads, ..., then a fixed tree), so the result does not depend on timing.
constexpr int FINISH_THREADS = 1024;
template <int K>
__global__ void __launch_bounds__(FINISH_THREADS) finish_sum_kernel(const double *partials,
                                                                    unsigned nblk, double *out) {
  __shared__ double sh[FINISH_THREADS][K];
  double acc[K];
  for (int k = 0; k < K; ++k) acc[k] = 0.0;
  for (unsigned b = blockIdx.x * FINISH_THREADS + threadIdx.x; b < nblk;
       b += gridDim.x * FINISH_THREADS)
    for (int k = 0; k < K; ++k) acc[k] += partials[size_t(b) * K + k];
  for (int k = 0; k < K; ++k) sh[threadIdx.x][k] = acc[k];
  __syncthreads();
  for (int s = FINISH_THREADS / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int k = 0; k < K; ++k) sh[threadIdx.x][k] += sh[threadIdx.x + s][k];
    __syncthreads();
  }
  if (threadIdx.x < K) out[blockIdx.x * K + threadIdx.x] = sh[0][threadIdx.x];
}

template <class Real>
__global__ void neighbors_kernel(const StepArgs<Real> a, int lattice, int32_t *src) {
  const unsigned n = blockIdx.x * BLOCK + threadIdx.x;
  const unsigned N = a.N;
  if (n >= N) return;
  const uint32_t link = a.link ? a.link[n] : 0u;
  const CellGeo g = cell_geo(n, a.nx, a.ny, a.nz);
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    int32_t v;
    if (link >> 31) {
      v = -1;
    } else {
      const int cls = lattice == 0 ? fluid_class_open<q>(g, link, a.f_wall, a.f_vel, a.f_press)
                                   : solute_class<q>(g, link, a.s_wall, a.s_inlet, a.s_outlet);
      v = cls == PULL_CELL ? int32_t((long long)n + src_delta<q>(g)) : -(1 + cls);
    }
    src[size_t(q) * N + n] = v;
  });
}

}  // namespace lbgb
