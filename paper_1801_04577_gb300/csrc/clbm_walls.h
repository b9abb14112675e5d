// The thermal wall rules (Eq. 26-28 and their off-midpoint form) and the
// arithmetic they and the collision are written in.  The step kernels take the
// rules as coefficients that the host makes from the functions below (the
// rules are linear in the temperatures along the link); the Nusselt reduction
// evaluates them directly.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstddef>
#include <cstdint>

namespace clbm {

// ---------------------------------------------------------------------------
// Arithmetic with the rounding points written out.  The same node update is
// compiled into several kernels (plane tiles, boundary nodes, batches, lattices
// resident in shared memory); left to itself the compiler contracts a * b + c
// differently in each, and a lattice would then depend on the kernel that
// advanced it.  With every multiply-add explicit they agree bit for bit.
// ---------------------------------------------------------------------------
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
#else
inline float fma_(float a, float b, float c) { return std::fma(a, b, c); }
inline double fma_(double a, double b, double c) { return std::fma(a, b, c); }
template <typename R> inline R mul_(R a, R b) { return a * b; }
template <typename R> inline R add_(R a, R b) { return a + b; }
template <typename R> inline R sub_(R a, R b) { return a - b; }
#endif
// ---------------------------------------------------------------------------
// Wall temperature (Eq. 28), one-sided when the second node is missing
// ---------------------------------------------------------------------------
template <typename R>
__host__ __device__ __forceinline__ R wall_temperature(R b1, R b2, R b3, R ne, R T1, R T2, bool have2) {
  const R n3 = mul_(ne, b3);
  if (have2)
    return fma_(mul_(R(9), b1), T1, fma_(R(3), n3, -mul_(b1, T2))) /
           fma_(R(8), b1, mul_(R(3), mul_(ne, b2)));
  return fma_(mul_(R(2), b1), T1, n3) / fma_(R(2), b1, mul_(ne, b2));
}

// Walls at the fraction q of a link (no counterpart in the paper; q = 1/2 is
// its half-way wall).  s = distance from the wall along the link into the
// fluid; the wall profile is the quadratic through (0, T_w), (q, T1),
// (1 + q, T2), i.e. q(1+q) dT/ds(0) = -(1+2q) T_w + (1+q)^2 T1 - q^2 T2, and
// dT/dn = -dT/ds(0) / (n.e).  T_w solves b1 dT/dn + b2 T_w = b3 (the line
// through (0, T_w), (q, T1) when T2 is missing).
template <typename R>
__host__ __device__ __forceinline__ R wall_temperature_q(R b1, R b2, R b3, R ne, R q, R T1, R T2, bool have2) {
  const R qn = mul_(q, ne);
  if (have2) {
    const R p = add_(R(1), q), qqn = mul_(qn, p);
    const R e = fma_(mul_(p, p), T1, -mul_(mul_(q, q), T2));
    return fma_(b1, e, mul_(b3, qqn)) / fma_(b1, fma_(R(2), q, R(1)), mul_(b2, qqn));
  }
  return fma_(b1, T1, mul_(b3, qn)) / fma_(b2, qn, b1);
}

// dT/dn at such a wall from the same profile.
template <typename R>
__host__ __device__ __forceinline__ R wall_gradient_q(R ne, R q, R Tw, R T1, R T2, bool have2) {
  if (have2) {
    const R p = R(1) + q;
    return ((R(1) + R(2) * q) * Tw - p * p * T1 + q * q * T2) / (q * p * ne);
  }
  return (Tw - T1) / (q * ne);
}

// The profile's value at the link midpoint s = q - 1/2, which Eq. 26 then
// imposes there.  q >= 1/2 or a wall with a flux term (b1 > 0): interpolation
// weights of the quadratic through the wall and the nodes at q and 1 + q.
// q < 1/2 at a Dirichlet wall: the quadratic through the wall and the nodes
// at 1 + q and 2 + q instead (bounded weights as q -> 0, none on the node's
// own T1, which would feed back into the node).  Both exact for quadratic
// profiles; lines through the available points in thin fluid layers.
template <typename R>
__host__ __device__ __forceinline__ R midpoint_temperature_q(R q, R Tw, R T1, R T2, bool have2, R T3,
                                                             bool have3, bool dirichlet) {
  const R m = fma_(R(2), q, R(-1));  // 2 (q - 1/2)
  const R p1 = add_(R(1), q);
  if (q >= R(0.5) || !dirichlet) {
    if (!have2) return fma_(sub_(T1, Tw), m / mul_(R(2), q), Tw);
    return fma_(R(3) / mul_(R(4), mul_(q, p1)), Tw,
                fma_(mul_(R(3), m) / mul_(R(4), q), T1, mul_(-(m / mul_(R(4), p1)), T2)));
  }
  if (have2 && have3) {
    const R p2 = add_(R(2), q);
    return fma_(R(15) / mul_(R(4), mul_(p1, p2)), Tw,
                fma_(mul_(R(5), m) / mul_(R(4), p1), T2, mul_(-(mul_(R(3), m) / mul_(R(4), p2)), T3)));
  }
  if (have2) return fma_(sub_(T2, Tw), m / mul_(R(2), p1), Tw);
  return Tw;
}

// A wall link's rule for the step: Eq. 26's cT2 (T_m - T0), with T_m the
// temperature at the link midpoint, as
//   k[0] s1 + k[1] s2 + k[3] s3 + k[2],   s = T - T0 + Q/2 at the nodes q, 1 + q, 2 + q from the wall.
// T_w is linear in (T1, T2) with the constant term from b3; T_m is a weighted
// sum of T_w, T1, T2, T3.
inline void link_heat(double b1, double b2, double b3, double ne, double q, bool have2, bool have3, double T0,
                      double hQ, double cT2, double (&k)[4]) {
  const bool mid = q == 0.5, dirichlet = b1 == 0.0;
  have3 = have3 && have2 && q < 0.5 && dirichlet;
  auto wall = [&](double b, double T1, double T2) {
    return mid ? wall_temperature(b1, b2, b, ne, T1, T2, have2) : wall_temperature_q(b1, b2, b, ne, q, T1, T2, have2);
  };
  auto weight = [&](double w, double T1, double T2, double T3) {
    return mid ? w : midpoint_temperature_q(q, w, T1, T2, have2, T3, have3, dirichlet);
  };
  const double w = weight(1, 0, 0, 0);  // of T_w
  // The weight on T1 is w b1 (...) + 3 (2q - 1) / 4q, two terms of order 1 / q whose
  // difference stays bounded as q -> 0: in closed form off the half-way wall.
  const double flux = b2 * ne, D = b1 * (1 + 2 * q) + flux * q * (1 + q);
  const double a = mid || (dirichlet && q < 0.5) ? w * wall(0.0, 1, 0) + weight(0, 1, 0, 0)
                   : have2 ? 0.75 * (b1 * (4 * q + 1) + (2 * q - 1) * (1 + q) * flux) / D
                           : (b1 + (q - 0.5) * flux) / (b1 + flux * q);
  const double b = have2 ? w * wall(0.0, 0, 1) + weight(0, 0, 1, 0) : 0.0;
  const double d = have3 ? weight(0, 0, 0, 1) : 0.0;
  k[0] = cT2 * a;
  k[1] = cT2 * b;
  k[3] = cT2 * d;
  k[2] = cT2 * (w * wall(b3, 0, 0) + (a + b + d) * (T0 - hQ) - T0);
}

// The same coefficients rounded to the compute type R.  A wall of given flux
// (b2 = 0) gives a uniform temperature back as much heat as it takes: its
// weights sum to the share of the heat that the collision keeps in an axis
// pair, cT2 but for the rounding of its constants (`share`, heat_share).
// Rounded one by one they miss it by about an ulp, always to the same side, a
// leak of 5e-8 (FP32) of T - T0 a link and step.  So the second is what the
// first leaves of it; |k[1]| <= cT2 / 4 holds the sum to a fraction of an ulp.
// T against FP64, geometric mean over 24 cavities (24^2 .. 128^2, Ra 1e3 .. 1e5)
// after 2000 / 8000 FP32 steps: 5.9e-8 / 2.9e-7 one by one, 6.7e-8 / 2.9e-7
// with a sum of (R)cT2, 4.2e-8 / 2.1e-7 so (rules evaluated by division at each
// link: 7.7e-8 / 3.4e-7).
template <typename R>
inline void round_heat(const double (&k)[4], double b2, double share, R (&o)[4]) {
  for (int m = 0; m < 4; ++m) o[m] = (R)k[m];
  if (b2 != 0.0) return;
  if (k[1] != 0.0)
    o[1] = (R)(share - (double)o[0]);  // (k[3] is zero where b1 > 0)
  else
    o[0] = (R)share;
}

// Bounce-back across a link as k[0] f_i + k[1] f_i(next node) + k[2] f_j, with
// f_i the population leaving towards the wall and f_j its reflection (Bouzidi,
// Firdaouss and Lallemand 2001; half-way: f_i).
inline void link_bounce(double q, bool have2, double (&k)[3]) {
  k[0] = 1.0;
  k[1] = k[2] = 0.0;
  if (q < 0.5 && have2) {
    k[0] = 2.0 * q;
    k[1] = 1.0 - 2.0 * q;
  } else if (q > 0.5) {
    k[0] = 1.0 / (2.0 * q);
    k[2] = (2.0 * q - 1.0) / (2.0 * q);
  }
}

// First coefficient of link `dir` of a node's entry `slot` in the tables of link_heat (dir 1..4) and
// link_bounce (dir 1..8); slots below kMaxLinkSlots.  Unsigned 32-bit numbers, the bounce's of its
// link: with the slot itself widened to 64 bits the boundary update takes up to 18 more registers
// (annulus 1024^2 FP32 16.3 -> 16.9 us a step), with the heat's link number 1021 x 509 BF16 takes
// 7.85 instead of 7.80.
constexpr int kMaxLinkSlots = 1 << 28;
__host__ __device__ constexpr uint32_t heat_entry(int slot, int dir) { return 16u * (uint32_t)slot + 4u * (uint32_t)(dir - 1); }
__host__ __device__ constexpr size_t bounce_entry(int slot, int dir) { return (size_t)(8u * (uint32_t)slot + (uint32_t)(dir - 1)) * 3; }

// The thermal rule of an axis link off the midpoint, q < 1/2, at a Dirichlet
// wall (b1 = 0) reads the third node x_f - 2 e_i: its row, for the link `dir`
// (1..4) of a node in row y.
inline bool reads_third(int dir, double q, double b1) { return dir <= 4 && q < 0.5 && b1 == 0.0; }
inline int third_row(int y, int dir) { return y - (dir == 2 ? 2 : dir == 4 ? -2 : 0); }

// Whether a slab that stores `ny` rows, its row y being row gy of a lattice of NY
// rows, holds that node's row (its ghost rows are whole copies), or there is none.
inline bool slab_holds_third(int y, int gy, int dir, int ny, int NY, bool py) {
  const int y3 = third_row(y, dir), gy3 = third_row(gy, dir);
  return (y3 >= 0 && y3 < ny) || (!py && (gy3 < 0 || gy3 >= NY));
}

// Whether the resident steps can evaluate that rule.  A band keeps one ghost
// row on either side, and of it only what streams across is kept up to date
// away from walls, so the third node must lie among the band's own rows.  Several
// bands: refused.  One band: all rows are its own, but across the seam of a
// periodic y axis the node would be a ghost row's or lie beyond it; beyond a wall
// there is no third node (link_heat's have3).
inline bool band_holds_third(int y, int dir, int ny, int cl, bool py) {
  const int y3 = third_row(y, dir);
  return cl == 1 && (!py || (y3 >= 0 && y3 < ny));
}

}  // namespace clbm
