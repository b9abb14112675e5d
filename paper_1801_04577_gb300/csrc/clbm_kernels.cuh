// Device code of the fused cascaded thermal LBM step for sm_103a.
//
// One time step per node, in one pass over HBM (pull scheme):
//   pull      f_i(x) = f*_i(x - e_i), g_i(x) = g*_i(x - e_i)      Eq. 11, Eq. 21
//   walls     half-way bounce-back for f (Sec. 3); general bounce-back for g
//             with T_w from Eq. 28                                  Eq. 26-28
//   macros    T = sum g + Q/2, F = F_v + rho0 g beta (T - T0) e_y,
//             rho = sum f, u = (sum f e + F/2)/rho                 Eq. 25, 2, 12
//   collide   central moments (Eq. 4-6), relaxation (Eq. 7-10),
//             back-transformation (text after Eq. 11)
//   thermal   Eq. 15-20 with the heat source of Eq. 23-24
//   store     f*(x), g*(x)
//
// Layout and precision.  The state kept in HBM is the post-collision pair
// (f*, g*) at time t, stored structure-of-arrays as deviations from the rest
// state, d_i = f*_i - w_i rho0 and h_i = g*_i - w^T_i T0.  The collision is
// rewritten in these deviations (the rest-state moments at velocity u are
// known in closed form), so every intermediate is a small number and FP32
// keeps its relative precision on the physically relevant part.
//
// Moment transforms.  The nine moments {0,1,2}^2 of Eq. 5 are a tensor
// product, so N(u) M f is computed as a 1-D central-moment transform along x
// for each of the three rows of velocities, then along y (and the inverse in
// the opposite order).  This is the same linear map as Eq. 6, evaluated with
// about a quarter of the operations; it relies on N(u)^-1 = N(-u).
//
// Vectorisation.  A warp owns 32*V consecutive nodes of one row; each lane
// loads V contiguous values of every plane with one 16-byte (8-byte for
// 16-bit storage) load.  The x-shift of the pull is done with one warp
// shuffle per plane; lanes 0 and 31 fetch the single value that crosses the
// warp boundary.  Box walls and periodic seams are selects of an address in the
// tiles (box_tile); nodes next to solids, and the edges of lattices with a mask
// or moving sides, are updated from a list of their own (node_update).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "clbm_internal.h"
#include "clbm_walls.h"

namespace clbm {

constexpr int kStepThreads = 128;
constexpr int kRedThreads = 256;

// ---------------------------------------------------------------------------
// Lattice (Eq. 3)
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int ex_of(int d) {
  return (d == 1 || d == 5 || d == 8) ? 1 : ((d == 3 || d == 6 || d == 7) ? -1 : 0);
}
__host__ __device__ constexpr int ey_of(int d) {
  return (d == 2 || d == 5 || d == 6) ? 1 : ((d == 4 || d == 7 || d == 8) ? -1 : 0);
}
__host__ __device__ constexpr int opp_of(int d) {
  return d == 0 ? 0 : (d <= 4 ? ((d + 1) % 4) + 1 : ((d - 5 + 2) % 4) + 5);
}

// ---------------------------------------------------------------------------
// Storage formats
// ---------------------------------------------------------------------------
template <typename S>
struct Traits;
template <>
struct Traits<double> {
  using R = double;
  static constexpr int V = 2;
};
template <>
struct Traits<float> {
  using R = float;
  static constexpr int V = 4;
};
template <>
struct Traits<__half> {
  using R = float;
  static constexpr int V = 4;
};
template <>
struct Traits<__nv_bfloat16> {
  using R = float;
  static constexpr int V = 4;
};

__device__ __forceinline__ double to_r(double v) { return v; }
__device__ __forceinline__ float to_r(float v) { return v; }
__device__ __forceinline__ float to_r(__half v) { return __half2float(v); }
__device__ __forceinline__ float to_r(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename S, typename R>
__device__ __forceinline__ S from_r(R v);
template <>
__device__ __forceinline__ double from_r<double, double>(double v) { return v; }
template <>
__device__ __forceinline__ float from_r<float, float>(float v) { return v; }
template <>
__device__ __forceinline__ __half from_r<__half, float>(float v) { return __float2half_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat16 from_r<__nv_bfloat16, float>(float v) {
  return __float2bfloat16_rn(v);
}

// Vector load / store of V consecutive elements as one naturally aligned
// access of V * sizeof(S) bytes (2 to 16 bytes).
template <int B>
struct RawOf;
template <>
struct RawOf<2> {
  using T = unsigned short;
};
template <>
struct RawOf<4> {
  using T = unsigned int;
};
template <>
struct RawOf<8> {
  using T = uint2;
};
template <>
struct RawOf<16> {
  using T = uint4;
};

template <typename S, int V, typename R>
__device__ __forceinline__ void ldv(const S* p, R (&o)[V]) {
  using Raw = typename RawOf<sizeof(S) * V>::T;
  const Raw r = *reinterpret_cast<const Raw*>(p);
  S e[V];
  memcpy(e, &r, sizeof(Raw));
#pragma unroll
  for (int k = 0; k < V; ++k) o[k] = to_r(e[k]);
}

template <typename S, int V, typename R>
__device__ __forceinline__ void stv(S* p, const R (&o)[V]) {
  using Raw = typename RawOf<sizeof(S) * V>::T;
  S e[V];
#pragma unroll
  for (int k = 0; k < V; ++k) e[k] = from_r<S, R>(o[k]);
  Raw r;
  memcpy(&r, e, sizeof(Raw));
  *reinterpret_cast<Raw*>(p) = r;
}

// ---------------------------------------------------------------------------
// Stochastic rounding of 16-bit stores.  Round-to-nearest storage of a state
// that changes little from step to step rounds the same way every step, and the
// bias accumulates; stochastic rounding makes each store unbiased.  The random
// bits come from a counter-based hash of (step, node, plane): the "lowbias32"
// integer mixer published by C. Wellons ("Prospecting for Hash Functions", 2018).
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

// Hardware stochastic rounding of two floats into a packed 16-bit pair
// (cvt.rs, Blackwell): `lo` lands in the low half (the first element in
// memory), `hi` in the high half; rbits supplies the random bits.
__device__ __forceinline__ uint32_t cvt_rs_f16x2(float lo, float hi, uint32_t rbits) {
  uint32_t d;
  asm("cvt.rs.satfinite.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
  return d;
}
__device__ __forceinline__ uint32_t cvt_rs_bf16x2(float lo, float hi, uint32_t rbits) {
  uint32_t d;
  asm("cvt.rs.satfinite.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
  return d;
}

template <typename S>
__device__ __forceinline__ uint32_t cvt_rs2(float lo, float hi, uint32_t r);
template <>
__device__ __forceinline__ uint32_t cvt_rs2<__half>(float lo, float hi, uint32_t r) {
  return cvt_rs_f16x2(lo, hi, r);
}
template <>
__device__ __forceinline__ uint32_t cvt_rs2<__nv_bfloat16>(float lo, float hi, uint32_t r) {
  return cvt_rs_bf16x2(lo, hi, r);
}

// Stochastically rounded store of V values (16-bit formats only).
template <typename S, int V>
__device__ __forceinline__ void stv_sr(S* p, const float (&o)[V], uint32_t r0, uint32_t r1, int sub) {
  static_assert(sizeof(S) == 2, "stochastic rounding applies to 16-bit storage");
  if constexpr (V == 1) {
    const uint32_t w = (sub & 2) ? r1 : r0;
    *reinterpret_cast<unsigned short*>(p) =
        (sub & 1) ? (unsigned short)(cvt_rs2<S>(0.0f, o[0], w) >> 16) : (unsigned short)(cvt_rs2<S>(o[0], 0.0f, w) & 0xFFFFu);
  } else if constexpr (V == 2) {
    *reinterpret_cast<unsigned int*>(p) = cvt_rs2<S>(o[0], o[1], (sub & 2) ? r1 : r0);
  } else {
    static_assert(V == 4, "16-bit tiles use 1, 2 or 4 nodes per lane");
    *reinterpret_cast<uint2*>(p) = make_uint2(cvt_rs2<S>(o[0], o[1], r0), cvt_rs2<S>(o[2], o[3], r1));
  }
}

// The random bits of a store depend on the step, the node and the plane only,
// whichever kernel updates the node: one key per group of four nodes x0 = x & ~3
// of a row (the full mixer of step and node), and per plane two words: one
// multiply-xorshift of the key plus a golden-ratio multiple of the plane, and one
// more multiply-xorshift of that word; word 0 rounds nodes x0, x0 + 1 (low, high
// half), word 1 nodes x0 + 2, x0 + 3.
__device__ __forceinline__ uint32_t sr_key(uint32_t seed, long long group_node) {
  return seed ^ mix32((uint32_t)group_node);
}
__device__ __forceinline__ void sr_words(uint32_t key, int q, uint32_t& r0, uint32_t& r1) {
  r0 = (key + 0x9E3779B9u * (uint32_t)(q + 1)) * 0x7feb352du;
  r0 ^= r0 >> 15;
  r1 = r0 * 0x846ca68bu;
  r1 ^= r1 >> 16;
}

// ---------------------------------------------------------------------------
// 1 / rho.  FP32: to within 2 ulp (hardware approximation), which the FP32
// parity bound leaves ample room for; FP64: the exact quotient.
__host__ __device__ __forceinline__ double rcp_(double v) { return 1.0 / v; }
__host__ __device__ __forceinline__ float rcp_(float v) {
#ifdef __CUDA_ARCH__
  return __fdividef(1.0f, v);
#else
  return 1.0f / v;
#endif
}

// ---------------------------------------------------------------------------
// Constants in the compute type
// ---------------------------------------------------------------------------
template <typename R>
struct Co {
  R rho0, T0;
  R rgb;   // rho0 * g beta
  R Fvx, Fvy, Q, hQ, cT2;
  R vhc;   // viscous source: Q_v = vhc (k~11^2 + (k~20 - k~02)^2 / 4) / rho^2
  CollideK<R> k;  // rates combined with the scalings of the relaxed form
};

template <typename R>
__host__ __device__ __forceinline__ Co<R> make_co(const DevCoef& c) {
  Co<R> o;
  if constexpr (std::is_same<R, float>::value) {  // rounded on the host
    o.k = c.kf;
    const CoefF32& f = c.f;
    o.rho0 = f.rho0;
    o.T0 = f.T0;
    o.rgb = f.rgb;
    o.Fvx = f.Fvx;
    o.Fvy = f.Fvy;
    o.Q = f.Q;
    o.hQ = f.hQ;
    o.cT2 = f.cT2;
    o.vhc = f.vhc;
  } else {
    o.k = c.kd;
    o.rho0 = (R)c.rho0;
    o.T0 = (R)c.T0;
    o.rgb = (R)(c.rho0 * c.gbeta);
    o.Fvx = (R)c.Fvx;
    o.Fvy = (R)c.Fvy;
    o.Q = (R)c.Q;
    o.hQ = (R)(0.5 * c.Q);
    o.cT2 = (R)c.cT2;
    // nu (D^2 + G^2) with G = -3 s_nu k~11/rho, D = -3 s_nu (k~20 - k~02)/(2 rho), nu = (1/s_nu - 1/2)/3
    o.vhc = (R)(c.vh ? 3.0 * c.s_nu * c.s_nu * (1.0 / c.s_nu - 0.5) : 0.0);
  }
  return o;
}

// ---------------------------------------------------------------------------
// 1-D central-moment transform over the velocities {-1, 0, +1} and back
// ---------------------------------------------------------------------------
// First and second order from the row's sum c0, difference s = a+ - a- and
// sum q = a+ + a-; n2u = -2 u, uu = u^2.
template <typename R>
__host__ __device__ __forceinline__ void fwd1p(R c0, R s, R q, R u, R n2u, R uu, R& c1, R& c2) {
  c1 = fma_(-u, c0, s);
  c2 = fma_(uu, c0, fma_(n2u, s, q));
}
// The same from the three populations.
template <typename R>
__host__ __device__ __forceinline__ void fwd1(R am, R a0, R ap, R u, R n2u, R uu, R& c0, R& c1, R& c2) {
  const R q = add_(ap, am), s = sub_(ap, am);
  c0 = add_(q, a0);
  fwd1p(c0, s, q, u, n2u, uu, c1, c2);
}
template <typename R>
__host__ __device__ __forceinline__ void inv1(R c0, R c1, R c2, R u, R& am, R& a0, R& ap) {
  const R r1 = c1 + u * c0;
  const R r2 = c2 + (u + u) * c1 + u * u * c0;
  a0 = c0 - r2;
  ap = R(0.5) * (r2 + r1);
  am = R(0.5) * (r2 - r1);
}
// inv1 from halved first- and second-order inputs, c1h = c1 / 2 and c2h =
// c2 / 2, with u2 = 2u, hu = u / 2, hu2 = u^2 / 2: h1 = r1 / 2 and h2 = r2 / 2
// come out directly, so the two halvings of inv1 are not needed.  Scaling by
// a power of two is exact, so the result is inv1's to rounding.
template <typename R>
__host__ __device__ __forceinline__ void inv1h(R c0, R c1h, R c2h, R u2, R hu, R hu2, R& am, R& a0,
                                               R& ap) {
  const R h1 = fma_(hu, c0, c1h);
  const R h2 = fma_(hu2, c0, fma_(u2, c1h, c2h));
  a0 = fma_(R(-2), h2, c0);
  ap = add_(h2, h1);
  am = sub_(h2, h1);
}

// ---------------------------------------------------------------------------
// Collision of one node, on deviations.  In: pre-collision deviations d, h.
// Out (in place): post-collision deviations.
// ---------------------------------------------------------------------------
// VH: add the viscous dissipation source Q_v (Sec. 3.2), read from the
// pre-collision non-equilibrium central moments; it is returned in qv.  The
// Boussinesq force uses T without Q_v/2 (Q_v needs u, which needs the force).
//
// The pipe that computes it bounds the FP64 step (an FP64 instruction holds a
// quarter of a multiprocessor for 64 cycles) and instruction issue the 16-bit
// ones, so what counts is the number of instructions: 153, every product that
// feeds a sum fused into it, half moments and constants combined on the host
// (170 as compiled from plain expressions; 2048 x 1024 FP64 775 -> 716 us a
// step, 4096 x 2048 FP16 1.02x, FP32 unchanged: bound by memory).  Each
// rounding is written out, so that every kernel gives the same bits.
template <typename R, bool VH = false>
__host__ __device__ __forceinline__ void collide(const Co<R>& c, R (&d)[9], R (&h)[5], R& qv) {
  const CollideK<R>& k = c.k;
  // Eq. 25 (T - T0 = sum h + Q/2) and half of the force of Eq. 2
  const R k20 = add_(h[1], h[3]), k02 = add_(h[2], h[4]);
  const R sh = add_(add_(h[0], k20), k02);
  const R dT = add_(sh, c.hQ);
  const R hFy = fma_(k.hrgb, dT, k.hFy);
  // Eq. 12 (sum_i w_i e_i = 0, so the rest state adds nothing to j), from the
  // sums and differences of each velocity row, which the x-pass below reuses
  const R ms = sub_(d[8], d[7]), mq = add_(d[8], d[7]);  // e_y = -1
  const R zs = sub_(d[1], d[3]), zq = add_(d[1], d[3]);  // e_y =  0
  const R ps = sub_(d[5], d[6]), pq = add_(d[5], d[6]);  // e_y = +1
  const R m0 = add_(mq, d[4]), z0 = add_(zq, d[0]), p0 = add_(pq, d[2]);
  const R yq = add_(p0, m0), jy = sub_(p0, m0);
  const R drho = add_(yq, z0);
  const R jx = add_(add_(ms, zs), ps);
  const R inv_rho = rcp_(add_(c.rho0, drho));
  const R ux = mul_(add_(jx, k.hFx), inv_rho);
  const R uy = mul_(add_(jy, hFy), inv_rho);
  const R ux2 = mul_(ux, ux), uy2 = mul_(uy, uy);
  const R n2ux = mul_(R(-2), ux), n2uy = mul_(R(-2), uy);

  // central moments of the deviations: x-pass per velocity row, then y-pass
  R xm1, xm2, xz1, xz2, xp1, xp2;
  fwd1p(m0, ms, mq, ux, n2ux, ux2, xm1, xm2);  // e_y = -1
  fwd1p(z0, zs, zq, ux, n2ux, ux2, xz1, xz2);  // e_y =  0
  fwd1p(p0, ps, pq, ux, n2ux, ux2, xp1, xp2);  // e_y = +1
  R b01, b02, b10, b11, b12, b20, b21, b22;
  fwd1p(drho, jy, yq, uy, n2uy, uy2, b01, b02);
  fwd1(xm1, xz1, xp1, uy, n2uy, uy2, b10, b11, b12);
  fwd1(xm2, xz2, xp2, uy, n2uy, uy2, b20, b21, b22);

  // Eq. 7-10, minus the rest-state moments rho0 kappa_m(ux) kappa_n(uy),
  // kappa = (1, -u, 1/3 + u^2).  Each post-collision moment D_mn is formed
  // scaled by 2^-[m > 0] 2^-[n > 0] (H_mn; exact scalings folded into the
  // rates), the form the back-transformation inv1h takes on both passes.
  const R third = R(1.0 / 3.0);
  const R H10 = fma_(R(0.5), b10, k.hFx);  // D10 / 2, D10 = b10 + Fx
  const R H01 = fma_(R(0.5), b01, hFy);    // D01 / 2, D01 = b01 + Fy
  // the (k~20, k~02) block: with a = k~ - its equilibrium (a20, a02 below),
  // D20 = k~20 - a20 + ((1 - s_b)(a20 + a02) + (1 - s_nu)(a20 - a02)) / 2, so
  // D20 / 2 = b20 / 2 + al a20 + be a02 and D02 / 2 = b02 / 2 + be a20 + al a02
  const R a20 = fma_(c.rho0, ux2, fma_(-third, drho, b20));
  const R a02 = fma_(c.rho0, uy2, fma_(-third, drho, b02));
  const R H20 = fma_(k.be, a02, fma_(k.al, a20, mul_(R(0.5), b20)));
  const R H02 = fma_(k.be, a20, fma_(k.al, a02, mul_(R(0.5), b02)));
  const R uxy = mul_(ux, uy);
  const R H11 = fma_(k.nsnur4, uxy, mul_(k.snu4, b11));  // D11 / 4
  const R tx = add_(third, ux2), ty = add_(third, uy2);
  const R H21 = fma_(k.s3f, hFy, fma_(k.s3r4, mul_(tx, uy), mul_(k.s3m4, b21)));  // D21 / 4
  const R H12 = fma_(k.s3r4, mul_(ux, ty), fma_(k.s3m4, b12, k.s3Fx));            // D12 / 4
  const R w22 = fma_(ux2, ty, mul_(third, uy2));  // (ux^2 + uy^2) / 3 + ux^2 uy^2
  const R H22 = fma_(k.ns4r4, w22, fma_(k.s4n, drho, mul_(k.s4m4, b22)));  // D22 / 4
  qv = R(0);
  if constexpr (VH) {
    const R k11 = fma_(c.rho0, uxy, b11);
    const R kd = fma_(c.rho0, sub_(ux2, uy2), sub_(b20, b02));
    const R k2 = fma_(mul_(R(0.25), kd), kd, mul_(k11, k11));
    qv = mul_(mul_(c.vhc, mul_(inv_rho, inv_rho)), k2);
  }

  // back-transformation: y-pass inverse per x-order (rows m = 1, 2 come out
  // halved, as the x-pass wants them), then x-pass inverse per row
  const R hux = mul_(R(0.5), ux), huy = mul_(R(0.5), uy);
  const R hux2 = mul_(R(0.5), ux2), huy2 = mul_(R(0.5), uy2);
  R ym0, yz0, yp0, ym1, yz1, yp1, ym2, yz2, yp2;
  inv1h(drho, H01, H02, -n2uy, huy, huy2, ym0, yz0, yp0);
  inv1h(H10, H11, H12, -n2uy, huy, huy2, ym1, yz1, yp1);
  inv1h(H20, H21, H22, -n2uy, huy, huy2, ym2, yz2, yp2);
  inv1h(ym0, ym1, ym2, -n2ux, hux, hux2, d[7], d[4], d[8]);
  inv1h(yz0, yz1, yz2, -n2ux, hux, hux2, d[3], d[0], d[1]);
  inv1h(yp0, yp1, yp2, -n2ux, hux, hux2, d[6], d[2], d[5]);

  // thermal (Eq. 15-20, 23-24) on deviations from w^T T0; kappa^T = (1, -u, cT2 + u^2)
  const R k10 = sub_(h[1], h[3]), k01 = sub_(h[2], h[4]);
  // (1 - l1)(k10 - ux sh) / 2 + l1 T0 ux / 2 = l1m2 k10 + ux (l1T2 - l1m2 sh)
  const R w1 = fma_(-k.l1m2, sh, k.l1T2);
  const R t20 = fma_(ux2, sh, fma_(n2ux, k10, k20));
  const R t02 = fma_(uy2, sh, fma_(n2uy, k01, k02));
  // post-collision thermal moments, first and second order halved (G = E / 2)
  // so that the back-transformation needs no halving of its own
  R E00, src2h;
  if constexpr (VH) {
    const R Qt = add_(c.Q, qv);
    E00 = add_(sh, Qt);
    src2h = fma_(k.srct2, fma_(R(0.5), Qt, sh), mul_(k.srcq2, Qt));  // Eq. 25 with the total source
  } else {
    E00 = add_(sh, c.Q);
    src2h = fma_(k.srct2, dT, k.srcQ);
  }
  const R G10 = fma_(ux, w1, mul_(k.l1m2, k10));
  const R G01 = fma_(uy, w1, mul_(k.l1m2, k01));
  const R G20 = fma_(k.l2m2, t20, fma_(k.nl2T2, ux2, src2h));
  const R G02 = fma_(k.l2m2, t02, fma_(k.nl2T2, uy2, src2h));
  const R q10 = fma_(hux, E00, G10), q01 = fma_(huy, E00, G01);  // halves of the raw moments
  const R q20 = fma_(hux2, E00, fma_(-n2ux, G10, G20));
  const R q02 = fma_(huy2, E00, fma_(-n2uy, G01, G02));
  h[0] = fma_(R(-2), add_(q20, q02), E00);
  h[1] = add_(q20, q10);
  h[3] = sub_(q20, q10);
  h[2] = add_(q02, q01);
  h[4] = sub_(q02, q01);
}

// (HK selects nothing: every storage type takes the same constants.  The host harness of the
// collision's tests names it.)
template <typename R, bool HK = true>
__host__ __device__ __forceinline__ void collide_any(const Co<R>& c, bool vh, R (&d)[9], R (&h)[5],
                                                     R& qv) {
  if (vh)
    collide<R, true>(c, d, h, qv);
  else
    collide<R, false>(c, d, h, qv);
}

// Pre-collision equilibrium deviations (central moments Eq. 9 and Eq. 19 minus
// the rest-state moments) at (rho, u, T).
template <typename R>
__host__ __device__ __forceinline__ void equilibrium(const Co<R>& c, R rho, R ux, R uy, R T, R (&d)[9],
                                            R (&h)[5]) {
  const R third = R(1.0 / 3.0);
  const R r0 = c.rho0, drho = rho - r0, ux2 = ux * ux, uy2 = uy * uy;
  const R E00 = drho, E10 = r0 * ux, E01 = r0 * uy;
  const R E20 = third * drho - r0 * ux2, E02 = third * drho - r0 * uy2;
  const R E11 = -r0 * ux * uy;
  const R E21 = r0 * (third + ux2) * uy, E12 = r0 * ux * (third + uy2);
  const R E22 = R(1.0 / 9.0) * drho - r0 * (third * (ux2 + uy2) + ux2 * uy2);
  R ym0, yz0, yp0, ym1, yz1, yp1, ym2, yz2, yp2;
  inv1(E00, E01, E02, uy, ym0, yz0, yp0);
  inv1(E10, E11, E12, uy, ym1, yz1, yp1);
  inv1(E20, E21, E22, uy, ym2, yz2, yp2);
  inv1(ym0, ym1, ym2, ux, d[7], d[4], d[8]);
  inv1(yz0, yz1, yz2, ux, d[3], d[0], d[1]);
  inv1(yp0, yp1, yp2, ux, d[6], d[2], d[5]);
  const R dT = T - c.T0;
  const R T0 = c.T0;
  const R e00 = dT, e10 = T0 * ux, e01 = T0 * uy;
  const R e20 = c.cT2 * dT - T0 * ux2, e02 = c.cT2 * dT - T0 * uy2;
  const R q10 = e10 + ux * e00, q01 = e01 + uy * e00;
  const R q20 = e20 + (ux + ux) * e10 + ux2 * e00;
  const R q02 = e02 + (uy + uy) * e01 + uy2 * e00;
  h[0] = e00 - q20 - q02;
  h[1] = R(0.5) * (q20 + q10);
  h[3] = R(0.5) * (q20 - q10);
  h[2] = R(0.5) * (q02 + q01);
  h[4] = R(0.5) * (q02 - q01);
}

// The stored state as the boundary nodes read it: planes in device memory ...
template <typename S>
struct PlaneSrc {
  using Idx = long long;
  static constexpr bool kShared = false;
  const S* __restrict__ p;
  long long plane;
  __device__ __forceinline__ S at(int q, long long i) const { return p[q * plane + i]; }
};
// ... or whole nodes in shared memory, ST values apart.
template <typename S, int ST>
struct NodeSrc {
  using Idx = int;
  static constexpr bool kShared = true;
  const S* p;
  __device__ __forceinline__ S at(int q, int i) const { return p[i * ST + q]; }
};

// T at a node from its post-collision thermal deviations: T = T0 + sum h* - Q/2,
// Q including the node's stored viscous source when that is enabled.
template <class Src, typename R, typename Idx>
__device__ __forceinline__ R node_T(const Src& src, Idx idx, const Co<R>& c) {
  R s = to_r(src.at(9, idx));
#pragma unroll
  for (int q = 10; q < 14; ++q) s += to_r(src.at(q, idx));
  R t = c.T0 + s - c.hQ;
  if (c.vhc != R(0)) t = fma_(R(-0.5), to_r(src.at(14, idx)), t);
  return t;
}

// T - T0 + Q/2 at a node (the wall rules' constants absorb T0 - Q/2).
template <class Src, typename R, typename Idx>
__device__ __forceinline__ R node_heat(const Src& src, Idx idx, const Co<R>& c) {
  R s = to_r(src.at(9, idx));
#pragma unroll
  for (int q = 10; q < 14; ++q) s = add_(s, to_r(src.at(q, idx)));
  if (c.vhc != R(0)) s = fma_(R(-0.5), to_r(src.at(14, idx)), s);
  return s;
}

// A pair of constants for the compute type (FP32 arithmetic has its own copies).
template <typename R>
__device__ __forceinline__ const R* side_wall(const DevGeom& g, int sd, bool have2) {
  if constexpr (std::is_same<R, float>::value)
    return g.side_kf[sd][have2 ? 1 : 0];
  else
    return g.side_k[sd][have2 ? 1 : 0];
}

// Eq. 26's cT2 (T_m - T0) at box side sd for the node `own` with `next` behind it.
template <class Src, typename R, typename Idx>
__device__ __forceinline__ R side_heat(const Src& src, const DevGeom& g, const Co<R>& c, int sd, bool have2,
                                       Idx own, Idx next) {
  const R* k = side_wall<R>(g, sd, have2);
  R e = k[2];
  if (k[1] != R(0)) e = fma_(k[1], node_heat(src, next, c), e);
  if (k[0] != R(0)) e = fma_(k[0], node_heat(src, own, c), e);
  return e;
}

// New state of node (x, y) next to a wall, a solid or a periodic seam: pull,
// bounce-back, Eq. 26-28, collision.  src: the stored state, indexed
// y * g.pitch + x; fl, slot: its flags and its entry of the link tables
// (masked lattices).
//
// What bounds this is the length of its dependent chain, not its bytes: a
// block of boundary nodes that took 3 us held up every small step.  So a
// population that comes from a wall is the opposite one of the node itself,
// chosen by its address (no branch), and the wall temperature, linear in the
// temperatures along the link, is three or four host-made coefficients (no
// division, no branch on the kind of wall).
template <class Src, bool MASK, typename R>
__device__ __forceinline__ void node_update(const DevGeom& g, const Co<R>& c, const Src& src, int x, int y,
                                            uint32_t fl, int slot, R (&d)[9], R (&h)[5], R& qv) {
  using Idx = typename Src::Idx;
  const Idx own = (Idx)y * g.pitch + x;
  const bool x_lo = x == 0, x_hi = x == g.nx - 1;
  const bool y_lo = y == g.ylo, y_hi = y == g.yhi - 1;
  d[0] = to_r(src.at(0, own));
  h[0] = to_r(src.at(9, own));
  uint32_t wall = MASK ? (fl & 0xFFu) : 0u;  // bit j - 1: population j comes from a wall ...
  uint32_t box = 0;                          // ... of the box
#pragma unroll
  for (int j = 1; j < 9; ++j) {
    const int ex = ex_of(j), ey = ey_of(j);
    const bool outx = ex > 0 ? x_lo : (ex < 0 ? x_hi : false);
    const bool outl = ey > 0 && y_lo, outh = ey < 0 && y_hi;
    if ((outx && !g.px) || (outl && g.ywlo) || (outh && g.ywhi)) box |= 1u << (j - 1);
  }
  wall |= box;
#pragma unroll
  for (int j = 1; j < 9; ++j) {
    const int ex = ex_of(j), ey = ey_of(j);
    int sx = x - ex, sy = y - ey;  // within the storage, around the seam, or unused (a wall)
    if (ex != 0 && g.px) sx = sx < 0 ? g.nx - 1 : (sx >= g.nx ? 0 : sx);
    if (ey != 0 && g.py) sy = sy < 0 ? g.ny - 1 : (sy >= g.ny ? 0 : sy);
    const bool w = (wall >> (j - 1)) & 1u;
    const Idx from = w ? own : (Idx)sy * g.pitch + sx;
    d[j] = to_r(src.at(w ? opp_of(j) : j, from));
    if (j < 5) h[j] = to_r(src.at(w ? 9 + opp_of(j) : 9 + j, from));
  }
  // the node one further along the link, x_f - e_i = x + e_j
  auto ahead = [&](int ex, int ey, int n) -> Idx {
    int x2 = x + n * ex, y2 = y + n * ey;
    if (g.px) x2 = x2 < 0 ? x2 + g.nx : (x2 >= g.nx ? x2 - g.nx : x2);
    if (g.py) y2 = y2 < 0 ? y2 + g.ny : (y2 >= g.ny ? y2 - g.ny : y2);
    return (Idx)y2 * g.pitch + x2;
  };
  if (wall & 0xFu) {
    const R s1 = node_heat(src, own, c);
    // Eq. 26 at the wall of direction j = b + 1
    auto rule = [&](int b, int ex, int ey) {
      R ka, kb, kc, kd = R(0);
      if ((box >> b) & 1u) {
        bool have2;
        if (MASK)
          have2 = !((fl >> (kFlagSecond + b)) & 1u);
        else
          have2 = ex != 0 ? g.nx > 1 : !(ey > 0 ? (y_hi && g.ywhi) : (y_lo && g.ywlo));
        const R* k = side_wall<R>(g, ex > 0 ? 0 : (ex < 0 ? 1 : (ey > 0 ? 2 : 3)), have2);
        ka = k[0];
        kb = k[1];
        kc = k[2];
      } else {
        const R* k = static_cast<const R*>(g.lk_t) + heat_entry(slot, ((b + 2) & 3) + 1);  // link opp(j)
        ka = __ldg(k);
        kb = __ldg(k + 1);
        kc = __ldg(k + 2);
        kd = __ldg(k + 3);
      }
      R e = kc;
      if (kd != R(0)) e = fma_(kd, node_heat(src, ahead(ex, ey, 2), c), e);
      if (kb != R(0)) e = fma_(kb, node_heat(src, ahead(ex, ey, 1), c), e);
      if (ka != R(0)) e = fma_(ka, s1, e);
      return e;
    };
    if constexpr (MASK && Src::kShared) {
      // one pass per wall of the node, whichever its direction, so that nodes with walls in
      // different directions share it (resident 200 x 100 channel 3.5 -> 2.9 us a step; from planes in
      // device memory the passes by direction are faster, annulus 1.69 -> 1.62 ms)
      for (uint32_t m = wall & 0xFu; m; m &= m - 1) {
        const int b = __ffs((int)m) - 1;
        const R e = rule(b, (b == 0) - (b == 2), (b == 1) - (b == 3));
#pragma unroll
        for (int j = 1; j < 5; ++j)
          if (j == b + 1) h[j] = sub_(e, h[j]);
      }
    } else {
#pragma unroll
      for (int j = 1; j < 5; ++j)
        if ((wall >> (j - 1)) & 1u) h[j] = sub_(rule(j - 1, ex_of(j), ey_of(j)), h[j]);
    }
  }
  if (MASK && (fl & kFlagOffMid)) {  // walls off the link midpoint: interpolated bounce-back
#pragma unroll
    for (int j = 1; j < 9; ++j) {
      if (!(((wall & ~box) >> (j - 1)) & 1u)) continue;
      const int i = opp_of(j);
      const R* k = static_cast<const R*>(g.lk_f) + bounce_entry(slot, i);
      const R k0 = __ldg(k), k1 = __ldg(k + 1), k2 = __ldg(k + 2);
      R v = mul_(k2, to_r(src.at(j, own)));
      if (k1 != R(0)) v = fma_(k1, to_r(src.at(i, ahead(ex_of(j), ey_of(j), 1))), v);
      d[j] = fma_(k0, d[j], v);
    }
  }
  if (g.moving && box) {
    // moving box sides (not in the paper; Ladd's bounce-back): the reflected
    // population gains -6 w_i rho0 (e_i . u_w), e_i = -e_j
#pragma unroll
    for (int j = 1; j < 9; ++j) {
      if (!((box >> (j - 1)) & 1u)) continue;
      const int ex = ex_of(j), ey = ey_of(j);
      const bool outx = ex > 0 ? x_lo : (ex < 0 ? x_hi : false);
      const int sd = (outx && !g.px) ? (ex > 0 ? 0 : 1) : (ey > 0 ? 2 : 3);
      R uwx, uwy;
      if constexpr (std::is_same<R, float>::value) {
        uwx = g.side_uf[sd][0];
        uwy = g.side_uf[sd][1];
      } else {
        uwx = (R)g.side_u[sd][0];
        uwy = (R)g.side_u[sd][1];
      }
      const R w6 = j <= 4 ? R(6.0 / 9.0) : R(6.0 / 36.0);
      d[j] = fma_(mul_(w6, c.rho0), add_(mul_(R(ex), uwx), mul_(R(ey), uwy)), d[j]);
    }
  }
  collide_any<R>(c, c.vhc != R(0), d, h, qv);
}

// ---------------------------------------------------------------------------
// The fused step kernel
// ---------------------------------------------------------------------------
// Store of one value (stochastically rounded for 16-bit storage when asked).
template <typename S, typename R>
__device__ __forceinline__ void st1(S* p, R v, int stochastic, uint32_t key, int q, int sub) {
  if constexpr (sizeof(S) == 2) {
    if (stochastic) {
      uint32_t r0, r1;
      sr_words(key, q, r0, r1);
      const float o[1] = {v};
      stv_sr<S, 1>(p, o, r0, r1, sub);
      return;
    }
  }
  *p = from_r<S, R>(v);
}

// Steps of more than one wave of blocks are launched as programmatic
// dependents: the next step's first blocks take the places that the last wave
// leaves, read their arguments, and wait here until the stores of the step
// before are visible (nothing before touches the state).  Per step: annulus
// 2048 FP32 79.9 -> 78.9 us, FP16 4096 x 2048 79.1 -> 78.6, 1024 x 512 FP32
// 8.65 -> 8.44.  In one wave the early blocks would land unevenly beside the
// running ones (FP64 101^2 9.0 -> 12.6 us): those steps are launched plainly.
__device__ __forceinline__ void step_wait() {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

// Interior update of lattices with a mask or moving sides.  One warp updates
// the 32 * V nodes x = xw .. xw + 32V - 1 of row y (each lane owns V consecutive
// nodes); all 32 lanes must call it together.  Every node is pulled and collided
// as if it were an interior fluid node: rows beyond a non-periodic edge are
// clamped and the ±1 x-shift at the row ends reads a neighbour, so what comes
// out for the first and last column (and, next to solids, for flagged nodes) is
// wrong.  Those nodes are the boundary list's: the tile leaves them out, or
// (MASKSTORE false) writes the flagged ones provisionally before a boundary
// launch replaces them.  Keeping the walls out keeps the warps free of divergent
// wall code.
template <typename S, int V, bool VH, bool SKIP_DEAD, bool MASKSTORE>
__device__ __forceinline__ void step_tile(const DevGeom& g, const Co<typename Traits<S>::R>& c,
                                          const S* __restrict__ src, S* __restrict__ dst, int y,
                                          int xw, int lane, uint32_t seed, int stochastic,
                                          bool mixed = false) {
  using R = typename Traits<S>::R;
  const int x0 = xw + lane * V;
  const long long plane = g.plane;

  int ym = y - 1, yp = y + 1;  // rows the e_y = +1 / -1 populations come from
  if (g.py) {
    ym = ym < 0 ? g.ny - 1 : ym;
    yp = yp >= g.ny ? 0 : yp;
  } else {
    ym = ym < 0 ? 0 : ym;
    yp = yp >= g.ny ? g.ny - 1 : yp;
  }
  const int xl = x0 > 0 ? x0 - 1 : 0;
  const int xr = x0 + V < g.pitch ? x0 + V : g.pitch - 1;
  // SKIP_DEAD: a lane wholly beyond the row (x0 >= nx: the pitch padding of
  // the last tile) neither loads nor stores; it still takes part in the
  // shuffles, and the only value it passes on (to node nx - 1 from x = nx)
  // belongs to the last column, which the boundary update recomputes.  (The
  // 16-bit single-lattice kernels leave it off: the extra live state costs
  // them register spills, more than the padding they would skip.)
  uint16_t fl[V];  // flags of the lane's nodes in a tile that holds flagged ones
#pragma unroll
  for (int k = 0; k < V; ++k) fl[k] = 0;
  bool solid = false;  // ... all of them solid: such a lane, too, neither loads nor stores
  if constexpr (MASKSTORE) {
    if (mixed) {
      using Raw = typename RawOf<2 * V>::T;
      const Raw r = *reinterpret_cast<const Raw*>(g.flags + (long long)y * g.pitch + x0);
      memcpy(fl, &r, sizeof(Raw));
      solid = true;
#pragma unroll
      for (int k = 0; k < V; ++k) solid = solid && (fl[k] & kFlagSolid);
    }
  }
  const bool live = !SKIP_DEAD || (x0 < g.nx && !solid);

  R v[14][V];
#pragma unroll
  for (int q = 0; q < 14; ++q) {
    const int dir = q < 9 ? q : q - 9;
    const int ex = ex_of(dir), ey = ey_of(dir);
    const int row = ey > 0 ? ym : (ey < 0 ? yp : y);
    const S* base = src + q * plane + (long long)row * g.pitch;
    R t[V];
    if (live) {
      ldv<S, V>(base + x0, t);
    } else {
#pragma unroll
      for (int k = 0; k < V; ++k) t[k] = R(0);
    }
    if (ex == 0) {
#pragma unroll
      for (int k = 0; k < V; ++k) v[q][k] = t[k];
    } else if (ex > 0) {  // value from x - 1
      R left = __shfl_up_sync(0xffffffffu, t[V - 1], 1);
      if (lane == 0) left = to_r(base[xl]);
      v[q][0] = left;
#pragma unroll
      for (int k = 1; k < V; ++k) v[q][k] = t[k - 1];
    } else {  // value from x + 1
      R right = __shfl_down_sync(0xffffffffu, t[0], 1);
      if (lane == 31 && live) right = to_r(base[xr]);
#pragma unroll
      for (int k = 0; k < V - 1; ++k) v[q][k] = t[k + 1];
      v[q][V - 1] = right;
    }
  }

  R qv[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    R d[9], h[5];
#pragma unroll
    for (int q = 0; q < 9; ++q) d[q] = v[q][k];
#pragma unroll
    for (int q = 0; q < 5; ++q) h[q] = v[9 + q][k];
    collide<R, VH>(c, d, h, qv[k]);
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q][k] = d[q];
#pragma unroll
    for (int q = 0; q < 5; ++q) v[9 + q][k] = h[q];
  }

  if (!live) return;
  S* out = dst + (long long)y * g.pitch + x0;
  if constexpr (MASKSTORE) {
    // a tile holding flagged nodes (solid, or fluid next to a wall) leaves them,
    // and the edge columns, to the boundary update of the same launch
    if (mixed) {
      uint32_t skip = 0;
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const int x = x0 + k;
        if (fl[k] != 0 || x == 0 || x == g.nx - 1) skip |= 1u << k;
      }
      if (skip) {
#pragma unroll
        for (int k = 0; k < V; ++k) {
          if ((skip >> k) & 1u) continue;
          const int x = x0 + k;
          if constexpr (VH) out[14 * plane + k] = from_r<S, R>(qv[k]);
          const uint32_t key = sr_key(seed, (long long)(y + g.yoff) * g.pitch + (x & ~3));
#pragma unroll
          for (int q = 0; q < 14; ++q) st1<S, R>(out + q * plane + k, v[q][k], stochastic, key, q, x & 3);
        }
        return;
      }
    }
  }
  if constexpr (VH) {  // the viscous source of this step, read back with T (15th plane)
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int x = x0 + k;
      if (x != 0 && x != g.nx - 1) out[14 * plane + k] = from_r<S, R>(qv[k]);
    }
  }
  // leave the first and last column to the boundary update running alongside
  if (x0 == 0 || (x0 <= g.nx - 1 && g.nx - 1 < x0 + V)) {
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int x = x0 + k;
      if (x == 0 || x == g.nx - 1) continue;
      const uint32_t key = sr_key(seed, (long long)(y + g.yoff) * g.pitch + (x & ~3));
#pragma unroll
      for (int q = 0; q < 14; ++q) st1<S, R>(out + q * plane + k, v[q][k], stochastic, key, q, x & 3);
    }
    return;
  }
  if constexpr (sizeof(S) == 2) {
    if (stochastic) {
      // x0 is a multiple of V (tiles start at multiples of 32 V nodes)
      const uint32_t key = sr_key(seed, (long long)(y + g.yoff) * g.pitch + (x0 & ~3));
#pragma unroll
      for (int q = 0; q < 14; ++q) {
        uint32_t r0, r1;
        sr_words(key, q, r0, r1);
        stv_sr<S, V>(out + q * plane, v[q], r0, r1, x0 & 3);
      }
      return;
    }
  }
#pragma unroll
  for (int q = 0; q < 14; ++q) stv<S, V>(out + q * plane, v[q]);
}

// Interior and walls in one: the tile for a lattice without a mask or moving
// sides, every node final.  The walls of a box need no list: a row next to a
// y wall pulls the opposite populations of its own row instead of the row
// beyond, and the lanes of the first and last column take the one value that
// an interior lane gets from the neighbouring tile from the opposite
// population of the edge node, or from around a periodic seam.
// EDGE: the tile touches a wall or seam.  It is a second copy of the code, and
// every choice in it is a select of an address or a value: a branch between
// the loads would keep them from being issued together (branches instead of
// selects took the FP32 4096 x 2048 step from 0.14 to 0.19 ms).
template <typename S, int V, bool VH, bool SKIP_DEAD, bool EDGE>
__device__ __forceinline__ void box_tile(const DevGeom& g, const Co<typename Traits<S>::R>& c,
                                            const S* __restrict__ src, S* __restrict__ dst, int y, int xw,
                                            int lane, uint32_t seed, int stochastic) {
  using R = typename Traits<S>::R;
  const int x0 = xw + lane * V;
  const long long plane = g.plane;
  const bool lo = EDGE && g.ywlo && y == g.ylo, hi = EDGE && g.ywhi && y == g.yhi - 1;
  int ym = y - 1, yp = y + 1;  // rows the e_y = +1 / -1 populations come from
  if (g.py) {
    ym = ym < 0 ? g.ny - 1 : ym;
    yp = yp >= g.ny ? 0 : yp;
  }
  const int lastx = g.nx - 1;
  const bool live = !SKIP_DEAD || x0 < g.nx;
  const bool first = EDGE && x0 == 0, last = EDGE && x0 <= lastx && lastx < x0 + V;
  const bool wall_l = first && !g.px, wall_r = last && !g.px;
  const long long row_y = (long long)y * g.pitch;
  // columns beyond the tile that lanes 0 and 31 (and the edge lanes) read: the
  // neighbouring tile's, the other end of a periodic row, the edge node's own
  const int xl = x0 > 0 ? x0 - 1 : (g.px ? lastx : 0);
  const int xr = last ? (g.px ? 0 : lastx) : (x0 + V < g.pitch ? x0 + V : g.pitch - 1);
  const bool get_l = lane == 0, get_r = (lane == 31 || last) && live;

  R v[14][V];
#pragma unroll
  for (int q = 0; q < 14; ++q) {
    const int dir = q < 9 ? q : q - 9, opp = q - dir + opp_of(dir);
    const int ex = ex_of(dir), ey = ey_of(dir);
    const bool w = ey > 0 ? lo : (ey < 0 ? hi : false);
    const int row = w ? y : (ey > 0 ? ym : (ey < 0 ? yp : y));
    const S* base = src + (w ? opp : q) * plane + (long long)row * g.pitch;
    R t[V];
    if (live) {
      ldv<S, V>(base + x0, t);
    } else {
#pragma unroll
      for (int k = 0; k < V; ++k) t[k] = R(0);
    }
    if (ex == 0) {
#pragma unroll
      for (int k = 0; k < V; ++k) v[q][k] = t[k];
    } else if (ex > 0) {  // value from x - 1
      const S* at = EDGE && wall_l ? src + opp * plane + row_y : base;
      R left = __shfl_up_sync(0xffffffffu, t[V - 1], 1);
      if (get_l) left = to_r(at[xl]);
      v[q][0] = w ? t[0] : left;
#pragma unroll
      for (int k = 1; k < V; ++k) v[q][k] = w ? t[k] : t[k - 1];
    } else {  // value from x + 1
      const S* at = EDGE && wall_r ? src + opp * plane + row_y : base;
      R right = __shfl_down_sync(0xffffffffu, t[0], 1);
      if (get_r) right = to_r(at[xr]);
      // the last column may lie inside the vector
#pragma unroll
      for (int k = 0; k < V - 1; ++k) v[q][k] = w ? t[k] : (EDGE && x0 + k == lastx ? right : t[k + 1]);
      v[q][V - 1] = w ? t[V - 1] : right;
    }
  }
  if (!g.px && (first || last)) {  // Eq. 26 at the x walls
    const PlaneSrc<S> ps{src, plane};
    if (first) v[10][0] = sub_(side_heat(ps, g, c, 0, g.nx > 1, row_y, row_y + 1), v[10][0]);
    if (last) {
      const R e = side_heat(ps, g, c, 1, g.nx > 1, row_y + lastx, row_y + lastx - 1);
#pragma unroll
      for (int k = 0; k < V; ++k)
        if (x0 + k == lastx) v[12][k] = sub_(e, v[12][k]);
    }
  }
  if ((lo || hi) && live) {  // rows next to a y wall: Eq. 26 for the whole row
    auto heat = [&](int row, R(&o)[V]) {
      const S* b = src + (long long)row * g.pitch + x0;
      R t[V];
      ldv<S, V>(b + 9 * plane, o);
#pragma unroll
      for (int q = 10; q < 14; ++q) {
        ldv<S, V>(b + q * plane, t);
#pragma unroll
        for (int k = 0; k < V; ++k) o[k] = add_(o[k], t[k]);
      }
      if (VH) {
        ldv<S, V>(b + 14 * plane, t);
#pragma unroll
        for (int k = 0; k < V; ++k) o[k] = fma_(R(-0.5), t[k], o[k]);
      }
    };
    auto wall = [&](int sd, int y2, bool have2, R(&h)[V]) {
      const R* k = side_wall<R>(g, sd, have2);
      R e[V], t[V];
#pragma unroll
      for (int m = 0; m < V; ++m) e[m] = k[2];
      if (k[1] != R(0)) {
        heat(y2, t);
#pragma unroll
        for (int m = 0; m < V; ++m) e[m] = fma_(k[1], t[m], e[m]);
      }
      if (k[0] != R(0)) {
        heat(y, t);
#pragma unroll
        for (int m = 0; m < V; ++m) e[m] = fma_(k[0], t[m], e[m]);
      }
#pragma unroll
      for (int m = 0; m < V; ++m) h[m] = sub_(e[m], h[m]);
    };
    if (lo) wall(2, y + 1, !hi, v[11]);
    if (hi) wall(3, y - 1, !lo, v[13]);
  }

  R qv[V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    R d[9], h[5];
#pragma unroll
    for (int q = 0; q < 9; ++q) d[q] = v[q][k];
#pragma unroll
    for (int q = 0; q < 5; ++q) h[q] = v[9 + q][k];
    collide<R, VH>(c, d, h, qv[k]);
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q][k] = d[q];
#pragma unroll
    for (int q = 0; q < 5; ++q) v[9 + q][k] = h[q];
  }
  if (!live) return;
  S* out = dst + row_y + x0;
  if constexpr (VH) stv<S, V>(out + 14 * plane, qv);
  if constexpr (sizeof(S) == 2) {
    if (stochastic) {
      // x0 is a multiple of V (tiles start at multiples of 32 V nodes)
      const uint32_t key = sr_key(seed, (long long)(y + g.yoff) * g.pitch + (x0 & ~3));
#pragma unroll
      for (int q = 0; q < 14; ++q) {
        uint32_t r0, r1;
        sr_words(key, q, r0, r1);
        stv_sr<S, V>(out + q * plane, v[q], r0, r1, x0 & 3);
      }
      return;
    }
  }
#pragma unroll
  for (int q = 0; q < 14; ++q) stv<S, V>(out + q * plane, v[q]);
}

// Boundary update of node index i (pitch layout).
template <typename S, bool MASK>
__device__ __forceinline__ void step_node(const DevGeom& g, const Co<typename Traits<S>::R>& c,
                                          const S* __restrict__ src, S* __restrict__ dst,
                                          long long i, uint32_t seed, int stochastic) {
  using R = typename Traits<S>::R;
  const int y = (int)(i / g.pitch), x = (int)(i - (long long)y * g.pitch);
  const long long plane = g.plane;
  R d[9], h[5], qv;
  const uint32_t fl = MASK ? (uint32_t)g.flags[i] : 0u;
  const int slot = MASK && (fl & kFlagLinks) ? g.slot[i] : 0;
  node_update<PlaneSrc<S>, MASK>(g, c, PlaneSrc<S>{src, plane}, x, y, fl, slot, d, h, qv);
  if (c.vhc != R(0)) dst[14 * plane + i] = from_r<S, R>(qv);
  // global node index of the group of four (the pitch is a multiple of 4)
  const uint32_t key = sr_key(seed, i + (long long)g.yoff * g.pitch - (x & 3));
#pragma unroll
  for (int q = 0; q < 14; ++q) st1<S, R>(dst + q * plane + i, q < 9 ? d[q] : h[q - 9], stochastic, key, q, x & 3);
}

// Stochastic-rounding key of a step: from the host value, or from the device
// step counter when the launch is part of a replayed graph.
__device__ __forceinline__ uint32_t step_seed(const StepArgs& a) {
  if (!a.stochastic) return 0u;
  if (!a.tdev) return a.seed;
  const long long t = *a.tdev + a.tstep;
  return (uint32_t)(t * 0x9E3779B1ull) ^ (uint32_t)(t >> 32);
}

// Blocks per SM the register budget is cut for: five (96 registers) where the
// step is memory-bound (FP32, FP64 storage); six (80 registers, a 44-byte
// spill) for 16-bit storage, which is bound by issue and memory latency and
// gains 2-6 % from the extra warps (measured A/B on one GB300).
template <typename S>
constexpr int kStepBlocks = sizeof(S) == 2 ? 6 : 5;

// Lattices without a mask or moving sides: blocks of up to four tiles of one
// row, in row order.  The row, and which copy of the tile runs, depend on
// blockIdx alone, so that the inner tiles keep their addresses in uniform
// registers (rows from threadIdx, or a choice per warp, cost the 16-bit step
// 15 %; edge tiles in blocks of their own, out of row order, the FP32 step 6 %).
// Without the boundary list's blocks a 4096 x 2048 step takes 132.7 us in FP32
// (135.0 with them; 14 planes in and out at the copy's rate: 138), 79.1 (80.0)
// in FP16, 87.4 (88.9) stochastic; 512 x 256 3.3 (4.9) in FP16; 101 x 101 FP64
// 9.0 (12.1).
template <typename S, int V, bool VH>
__global__ void __launch_bounds__(kStepThreads, kStepBlocks<S>) step_box_kernel(const StepArgs a, int xblocks,
                                                                              int rows) {
  using R = typename Traits<S>::R;
  const Co<R> c = make_co<R>(a.c);
  const S* src = static_cast<const S*>(a.src);
  S* dst = static_cast<S*>(a.dst);
  step_wait();
  const int b = blockIdx.x, row = b / xblocks, xb = b - row * xblocks;
  const int xw = (xb * blockDim.x + (threadIdx.x & ~31)) * V;
  if (xw >= a.g.nx) return;  // whole warps only
  const int y = a.g.ylo + (a.reverse ? rows - 1 - row : row);
  const bool edge = xb == 0 || xb == xblocks - 1 || (a.g.ywlo && y == a.g.ylo) || (a.g.ywhi && y == a.g.yhi - 1);
  if (edge)
    box_tile<S, V, VH, sizeof(S) != 2, true>(a.g, c, src, dst, y, xw, threadIdx.x & 31, step_seed(a), a.stochastic);
  else
    box_tile<S, V, VH, sizeof(S) != 2, false>(a.g, c, src, dst, y, xw, threadIdx.x & 31, step_seed(a), a.stochastic);
}

// Lattices with a mask or moving sides: interior and boundary nodes are
// disjoint, so one launch does both.  The first nbb blocks update the boundary
// list; the others are interior tiles, which leave those nodes out.  The
// latency-bound boundary work then overlaps the streaming interior work
// instead of following it.
template <typename S, bool VH, bool MASKED>
__global__ void __launch_bounds__(kStepThreads, kStepBlocks<S>) step_fused_kernel(const StepArgs a, int nbb,
                                                                                int xblocks, int y0, int rows) {
  using R = typename Traits<S>::R;
  constexpr int V = Traits<S>::V;
  const Co<R> c = make_co<R>(a.c);
  step_wait();
  if ((int)blockIdx.x < nbb) {
    const int k = blockIdx.x * kStepThreads + threadIdx.x;
    if (k < a.nb)
      step_node<S, MASKED>(a.g, c, static_cast<const S*>(a.src), static_cast<S*>(a.dst), a.bnodes[k],
                           step_seed(a), a.stochastic);
    return;
  }
  const int b = blockIdx.x - nbb;
  const int row = b / xblocks;
  const int y = y0 + (a.reverse ? rows - 1 - row : row);
  const int lane = threadIdx.x & 31;
  const int warp = (b % xblocks) * (kStepThreads / 32) + (threadIdx.x >> 5);
  const int xw = warp * 32 * V;
  if (xw >= a.g.nx) return;  // whole warps only
  if constexpr (MASKED) {  // tile classes: 0 no fluid, 1 unflagged fluid, 2 holds flagged nodes
    const uint8_t cls = a.g.tile_fluid[(long long)y * a.g.tiles_per_row + warp];
    if (!cls) return;
    step_tile<S, V, VH, sizeof(S) != 2, true>(a.g, c, static_cast<const S*>(a.src), static_cast<S*>(a.dst), y, xw, lane,
                                              step_seed(a), a.stochastic, cls == 2);
  } else {
    step_tile<S, V, VH, sizeof(S) != 2, false>(a.g, c, static_cast<const S*>(a.src), static_cast<S*>(a.dst), y, xw, lane,
                                               step_seed(a), a.stochastic);
  }
}

// ---------------------------------------------------------------------------
// Initialisation: equilibrium at the given fields, then one collision (the
// stored state is post-collision).
// ---------------------------------------------------------------------------
template <typename S>
__global__ void init_kernel(const DevGeom g, const DevCoef cf, S* __restrict__ dst,
                            const double* __restrict__ rho, const double* __restrict__ ux,
                            const double* __restrict__ uy, const double* __restrict__ T) {
  using R = typename Traits<S>::R;
  const Co<R> c = make_co<R>(cf);
  // one thread per column of the padded rows (every stored row, ghost rows too)
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.pitch) return;
  for (int y = (int)blockIdx.y; y < g.ny; y += (int)gridDim.y) {
    const long long i = (long long)y * g.pitch + x;
    R d[9], h[5];
    bool active = x < g.nx && y >= g.ylo && y < g.yhi;  // own rows (ghost rows: zero until exchanged)
    if (g.flags) active = active && !(g.flags[i] & kFlagSolid);
    if (active) {
      const long long k = (long long)(y - g.ylo) * g.nx + x;
      const R r = rho ? (R)rho[k] : c.rho0;
      const R u = ux ? (R)ux[k] : R(0);
      const R w = uy ? (R)uy[k] : R(0);
      const R t = T ? (R)T[k] : c.T0;
      equilibrium(c, r, u, w, t, d, h);
      R qv;
      collide_any<R>(c, cf.vh != 0, d, h, qv);
      if (cf.vh) dst[14 * g.plane + i] = from_r<S, R>(qv);
    } else {
      if (cf.vh) dst[14 * g.plane + i] = from_r<S, R>(R(0));
#pragma unroll
      for (int q = 0; q < 9; ++q) d[q] = R(0);
#pragma unroll
      for (int q = 0; q < 5; ++q) h[q] = R(0);
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) dst[q * g.plane + i] = from_r<S, R>(d[q]);
#pragma unroll
    for (int q = 0; q < 5; ++q) dst[(9 + q) * g.plane + i] = from_r<S, R>(h[q]);
  }
}

// ---------------------------------------------------------------------------
// Macroscopic fields from a post-collision state, in FP64:
//   rho = rho0 + sum d*, T = T0 + sum h* - Q/2, u = (sum d* e - F/2)/rho
// (the collision adds F to the first moments and Q to the zeroth thermal one).
// ---------------------------------------------------------------------------
template <typename S>
__device__ __forceinline__ void node_macros(const DevCoef& c, const S* __restrict__ b,
                                            long long plane, long long i, double& rho, double& ux,
                                            double& uy, double& T) {
  double f[9], s = 0.0;
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = (double)to_r(b[q * plane + i]);
#pragma unroll
  for (int q = 9; q < 14; ++q) s += (double)to_r(b[q * plane + i]);
  const double qv = c.vh ? (double)to_r(b[14 * plane + i]) : 0.0;
  T = c.T0 + s - 0.5 * (c.Q + qv);
  // the Boussinesq force uses T without the viscous source's half
  const double Fx = c.Fvx, Fy = c.Fvy + c.rho0 * c.gbeta * (T - 0.5 * qv - c.T0);
  const double dr = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  rho = c.rho0 + dr;
  const double jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
  const double jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  ux = (jx - 0.5 * Fx) / rho;
  uy = (jy - 0.5 * Fy) / rho;
}

// The same in the collision's arithmetic R (FP32 below FP64 storage).
template <typename S, typename R>
__device__ __forceinline__ void node_macros_r(const Co<R>& c, bool vh, const S* __restrict__ b,
                                              long long plane, long long i, R& rho, R& ux, R& uy,
                                              R& T) {
  R f[9], s = R(0);
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = (R)to_r(b[q * plane + i]);
#pragma unroll
  for (int q = 9; q < 14; ++q) s += (R)to_r(b[q * plane + i]);
  const R qv = vh ? (R)to_r(b[14 * plane + i]) : R(0);
  T = c.T0 + s - R(0.5) * (c.Q + qv);
  const R Fx = c.Fvx, Fy = c.Fvy + c.rgb * (T - R(0.5) * qv - c.T0);
  const R dr = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  rho = c.rho0 + dr;
  const R jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
  const R jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  const R inv = R(1) / rho;
  ux = (jx - R(0.5) * Fx) * inv;
  uy = (jy - R(0.5) * Fy) * inv;
}

// Sums of one node's stored deviations in the arithmetic R: the zeroth and
// first moments of d*, the zeroth moment of h* and the viscous source slot.
template <typename R>
struct NodeSums {
  R dr, jx, jy, s, qv;
};

template <typename R, typename S>
__device__ __forceinline__ NodeSums<R> node_sums(const S* __restrict__ b, long long plane,
                                                 long long i, bool vh) {
  R f[9];
  NodeSums<R> o;
  o.s = R(0);
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = (R)to_r(b[q * plane + i]);
#pragma unroll
  for (int q = 9; q < 14; ++q) o.s += (R)to_r(b[q * plane + i]);
  o.qv = vh ? (R)to_r(b[14 * plane + i]) : R(0);
  o.dr = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  o.jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
  o.jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  return o;
}

// The reported fields of one fluid node.  FP64 storage: all in FP64.  Below
// it the sums and the velocity take the collision's FP32 arithmetic (the
// precision the state carries) and only the offsets rho0 and T0 are added in
// FP64, so that the deviations of rho and T keep every bit the sums have.
// Fy uses T - qv/2 - T0 = sum h* - Q/2 - qv, without the cancellation of T0.
template <typename S>
__device__ __forceinline__ void node_fields(const DevCoef& c, const Co<typename Traits<S>::R>& co,
                                            const S* __restrict__ b, long long plane, long long i,
                                            double& rho, double& ux, double& uy, double& T) {
  using R = typename Traits<S>::R;
  if constexpr (std::is_same<R, double>::value) {
    node_macros(c, b, plane, i, rho, ux, uy, T);
  } else {
    const NodeSums<R> n = node_sums<R>(b, plane, i, c.vh != 0);
    const R Fy = co.Fvy + co.rgb * (n.s - R(0.5) * co.Q - n.qv);
    const R inv = R(1) / (co.rho0 + n.dr);
    ux = (double)((n.jx - R(0.5) * co.Fvx) * inv);
    uy = (double)((n.jy - R(0.5) * Fy) * inv);
    rho = c.rho0 + (double)n.dr;
    T = c.T0 + (double)(n.s - R(0.5) * (co.Q + n.qv));
  }
}

// One thread per column x of the own rows; the rows are strided over gridDim.y.
template <typename S>
__global__ void moments_kernel(const DevGeom g, const DevCoef c, const S* __restrict__ b,
                               double* __restrict__ rho, double* __restrict__ ux,
                               double* __restrict__ uy, double* __restrict__ T) {
  using R = typename Traits<S>::R;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.nx) return;
  const Co<R> co = make_co<R>(c);
  for (int y = g.ylo + (int)blockIdx.y; y < g.yhi; y += (int)gridDim.y) {
    const long long i = (long long)y * g.pitch + x;
    const long long k = (long long)(y - g.ylo) * g.nx + x;  // own-row index
    double r = 0, u = 0, v = 0, t = 0;
    if (!g.flags || !(g.flags[i] & kFlagSolid)) node_fields<S>(c, co, b, g.plane, i, r, u, v, t);
    if (rho) rho[k] = r;
    if (ux) ux[k] = u;
    if (uy) uy[k] = v;
    if (T) T[k] = t;
  }
}

// ---------------------------------------------------------------------------
// Deterministic FP64 reductions: each block writes its partial sums; a single
// block adds the partials in index order.
// ---------------------------------------------------------------------------

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

template <int W>
__device__ __forceinline__ void block_sum_store(double (&acc)[W], double* out) {
  __shared__ double sh[kRedThreads / 32][W];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const double s = warp_sum(acc[k]);
    if (lane == 0) sh[wid][k] = s;
  }
  __syncthreads();
  if (threadIdx.x < W) {
    double s = 0.0;
    for (int w = 0; w < kRedThreads / 32; ++w) s += sh[w][threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// Squared one-step changes and squares of T, ux, uy at one fluid node, added
// to a[0..5] (a[6] counts a non-finite field).  FP64 storage: the fields of
// both states in FP64 and their differences.  Below it, in FP32 from the
// differences of the stored values, which are exact where the state barely
// moves (the differences of FP32 fields near rho0 and T0 would be rounded to
// their ulp):
//   dT = sum dh* - dqv/2,  du = (da - u(t-1) d(drho)) / rho(t),
// a = j - F/2 with dFy = rgb (sum dh* - dqv) (a(t) = a(t-1) + da, rho(t) =
// rho(t-1) + d(drho)).  Fields beyond ~1e19 overflow the FP32 squares and
// count as unstable, as a non-finite field does.
template <typename S, typename R>
__device__ __forceinline__ void residual_terms(const DevCoef& c, const Co<R>& co,
                                               const S* __restrict__ cur,
                                               const S* __restrict__ prev, long long plane,
                                               long long i, R (&a)[7]) {
  if constexpr (std::is_same<R, double>::value) {
    double r1, u1, v1, t1, r0, u0, v0, t0;
    node_macros(c, cur, plane, i, r1, u1, v1, t1);
    node_macros(c, prev, plane, i, r0, u0, v0, t0);
    a[0] += (t1 - t0) * (t1 - t0);
    a[1] += t1 * t1;
    a[2] += (u1 - u0) * (u1 - u0);
    a[3] += u1 * u1;
    a[4] += (v1 - v0) * (v1 - v0);
    a[5] += v1 * v1;
    if (!isfinite(r1) || !isfinite(u1) || !isfinite(v1) || !isfinite(t1)) a[6] += 1.0;
  } else {
    const bool vh = c.vh != 0;
    R f1[9], f0[9], df[9], s1 = R(0), s0 = R(0), ds = R(0);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      f1[q] = (R)to_r(cur[q * plane + i]);
      f0[q] = (R)to_r(prev[q * plane + i]);
      df[q] = f1[q] - f0[q];
    }
#pragma unroll
    for (int q = 9; q < 14; ++q) {
      const R h1 = (R)to_r(cur[q * plane + i]), h0 = (R)to_r(prev[q * plane + i]);
      s1 += h1;
      s0 += h0;
      ds += h1 - h0;
    }
    const R q1 = vh ? (R)to_r(cur[14 * plane + i]) : R(0);
    const R q0 = vh ? (R)to_r(prev[14 * plane + i]) : R(0);
    auto zeroth = [](const R* f) {
      return ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    };
    auto first_x = [](const R* f) { return (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]); };
    auto first_y = [](const R* f) { return (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]); };
    const R dq = q1 - q0;
    const R t1 = co.T0 + (s1 - R(0.5) * (co.Q + q1));
    const R dT = ds - R(0.5) * dq;
    const R Fy1 = co.Fvy + co.rgb * (s1 - R(0.5) * co.Q - q1);
    const R Fy0 = co.Fvy + co.rgb * (s0 - R(0.5) * co.Q - q0);
    const R rho1 = co.rho0 + zeroth(f1), rho0 = co.rho0 + zeroth(f0), ddr = zeroth(df);
    const R inv1 = R(1) / rho1, inv0 = R(1) / rho0;
    const R u1 = (first_x(f1) - R(0.5) * co.Fvx) * inv1;
    const R v1 = (first_y(f1) - R(0.5) * Fy1) * inv1;
    const R u0 = (first_x(f0) - R(0.5) * co.Fvx) * inv0;
    const R v0 = (first_y(f0) - R(0.5) * Fy0) * inv0;
    const R dax = first_x(df), day = first_y(df) - R(0.5) * co.rgb * (ds - dq);
    const R du = (dax - u0 * ddr) * inv1, dv = (day - v0 * ddr) * inv1;
    a[0] += dT * dT;
    a[1] += t1 * t1;
    a[2] += du * du;
    a[3] += u1 * u1;
    a[4] += dv * dv;
    a[5] += v1 * v1;
    if (!isfinite(rho1) || !isfinite(u1) || !isfinite(v1) || !isfinite(t1)) a[6] += R(1);
  }
}

// Work items are (own row, span of kRedThreads * kResV columns); a thread
// sums its kResV nodes of an item in R and adds that to its FP64 sums.  The
// items' partial sums depend on the row and columns alone, so slabs of one
// lattice add the same numbers (in another order).
constexpr int kResV = 8;

template <typename S>
__global__ void __launch_bounds__(kRedThreads)
    residual_kernel(const DevGeom g, const DevCoef c, const S* __restrict__ cur,
                    const S* __restrict__ prev, double* __restrict__ partials) {
  using R = typename Traits<S>::R;
  const Co<R> co = make_co<R>(c);
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  constexpr int span = kRedThreads * kResV;
  const int xch = (g.nx + span - 1) / span;
  const long long items = (long long)(g.yhi - g.ylo) * xch;
  for (long long it = blockIdx.x; it < items; it += gridDim.x) {
    const int yr = (int)(it / xch);
    const int x0 = (int)(it - (long long)yr * xch) * span + (int)threadIdx.x;
    const long long row = (long long)(yr + g.ylo) * g.pitch;
    R a[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < kResV; ++j) {
      const int x = x0 + j * kRedThreads;
      if (x < g.nx && !(g.flags && (g.flags[row + x] & kFlagSolid)))
        residual_terms<S, R>(c, co, cur, prev, g.plane, row + x, a);
    }
#pragma unroll
    for (int q = 0; q < 7; ++q) acc[q] += (double)a[q];
  }
  block_sum_store<8>(acc, partials + 8 * blockIdx.x);
}

// Conservation sums over the fluid nodes of the stored post-collision
// deviations, accumulated in FP64: Sum_i d_i, Sum_i d_i e_ix, Sum_i d_i e_iy,
// Sum_j h_j, the fluid-node count and the count of non-finite values.
template <typename S>
__global__ void __launch_bounds__(kRedThreads)
    totals_kernel(const DevGeom g, const S* __restrict__ b, double* __restrict__ partials) {
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const long long n = (long long)(g.yhi - g.ylo) * g.nx;  // own rows
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const int yl = (int)(k / g.nx), x = (int)(k - (long long)yl * g.nx);
    const long long i = (long long)(yl + g.ylo) * g.pitch + x;
    if (g.flags && (g.flags[i] & kFlagSolid)) continue;
    double f[9], s = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) f[q] = (double)to_r(b[q * g.plane + i]);
#pragma unroll
    for (int q = 9; q < 14; ++q) s += (double)to_r(b[q * g.plane + i]);
    const double m = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    const double jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
    const double jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    acc[0] += m;
    acc[1] += jx;
    acc[2] += jy;
    acc[3] += s;
    acc[4] += 1.0;
    if (!isfinite(m) || !isfinite(jx) || !isfinite(jy) || !isfinite(s)) acc[5] += 1.0;
  }
  block_sum_store<8>(acc, partials + 8 * blockIdx.x);
}

template <typename S>
__global__ void __launch_bounds__(kRedThreads)
    nusselt_kernel(const DevGeom g, const DevCoef c, const S* __restrict__ b,
                   const NuLink* __restrict__ links, int nlinks, double* __restrict__ partials) {
  double acc[2] = {0, 0};
  const Co<double> cd = make_co<double>(c);
  const PlaneSrc<S> src{b, g.plane};
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < nlinks; l += gridDim.x * blockDim.x) {
    const NuLink L = links[l];
    const double T1 = node_T(src, L.own, cd);
    const bool have2 = L.second >= 0;
    const double T2 = have2 ? node_T(src, L.second, cd) : 0.0;
    double grad;
    if (L.q == 0.5) {
      const double Tw = wall_temperature(L.b1, L.b2, L.b3, L.ne, T1, T2, have2);
      grad = have2 ? (8.0 * Tw - 9.0 * T1 + T2) / (3.0 * L.ne)  // Eq. 27
                   : (Tw - T1) / (0.5 * L.ne);
    } else {  // wall off the link midpoint
      const double Tw = wall_temperature_q(L.b1, L.b2, L.b3, L.ne, L.q, T1, T2, have2);
      grad = wall_gradient_q(L.ne, L.q, Tw, T1, T2, have2);
    }
    acc[0] += grad;
    acc[1] += isfinite(grad) ? 0.0 : 1.0;
  }
  block_sum_store<2>(acc, partials + 2 * blockIdx.x);
}

// ---------------------------------------------------------------------------
// Batched solves: the step kernel walks a tile list with a persistent grid
// (each warp takes tiles w, w + #warps, ...), so the same launch serves any
// number of active lattices; the list is rebuilt on the device as lattices
// converge.
// ---------------------------------------------------------------------------
// Each warp takes one contiguous chunk of the tile list (tiles are ordered by
// lattice, row, x), so it stays on one lattice for many tiles; the lattice's
// descriptor is copied into a per-warp shared-memory slot when it changes and
// read from there, instead of chasing it through global memory on every tile.
// MASKED: tiles cover only the rows that are not boundary rows and skip the
// first and last column: those nodes belong to the boundary launch that
// follows.  Otherwise every node is final (box_tile), and the lattice's
// constants are read from shared memory where they are used, which leaves
// registers for five blocks a multiprocessor where the step is not bound by
// memory alone (64 cavities of 32 .. 512: FP32 202 -> 185 us a step, with five
// blocks 201; FP16 179 -> 156 us, with four blocks 168).
template <typename S, int V, bool MASKED>
constexpr int kBatchBlocks = MASKED || sizeof(S) == 8 || (V == Traits<S>::V && sizeof(S) == 4) ? 4 : 5;

template <typename S, int V, bool MASKED>
__global__ void __launch_bounds__(kStepThreads, (kBatchBlocks<S, V, MASKED>))
    batch_step_kernel(const BatchLat* __restrict__ lats, const int4* __restrict__ tiles,
                      const int* __restrict__ count, int parity, const long long* __restrict__ tptr,
                      int tstep, int stochastic) {
  using R = typename Traits<S>::R;
  static_assert(sizeof(BatchLat) % 8 == 0, "descriptor is copied in 8-byte words");
  __shared__ BatchLat slot[kStepThreads / 32];
  __shared__ Co<R> coef[MASKED ? 1 : kStepThreads / 32];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const long long n = *count;
  const long long nw = (long long)gridDim.x * (kStepThreads / 32);
  const long long chunk = (n + nw - 1) / nw;
  const long long begin = ((long long)blockIdx.x * (kStepThreads / 32) + wib) * chunk;
  const long long end = begin + chunk < n ? begin + chunk : n;
  uint32_t seed = 0;
  if (stochastic) {
    const long long t = *tptr + tstep;
    seed = (uint32_t)(t * 0x9E3779B1ull) ^ (uint32_t)(t >> 32);
  }
  BatchLat& L = slot[wib];
  int cur = -1;
  Co<R> c;
  for (long long w = begin; w < end; ++w) {
    const int4 tl = tiles[w];
    if (tl.x != cur) {
      __syncwarp();
      const unsigned long long* from = reinterpret_cast<const unsigned long long*>(lats + tl.x);
      unsigned long long* to = reinterpret_cast<unsigned long long*>(&L);
      for (int k = lane; k < (int)(sizeof(BatchLat) / 8); k += 32) to[k] = from[k];
      __syncwarp();
      cur = tl.x;
      if constexpr (MASKED) {
        c = make_co<R>(L.c);
      } else {
        if (lane == 0) coef[wib] = make_co<R>(L.c);
        __syncwarp();
      }
    }
    const S* src = static_cast<const S*>(L.buf[parity]);
    S* dst = static_cast<S*>(L.buf[parity ^ 1]);
    if constexpr (MASKED) {
      step_tile<S, V, false, true, false>(L.g, c, src, dst, tl.y, tl.z, lane, seed, stochastic);
    } else {
      // one copy of the tile: rows of a few hundred nodes are mostly edge tiles anyway
      box_tile<S, V, false, true, true>(L.g, coef[wib], src, dst, tl.y, tl.z, lane, seed, stochastic);
    }
  }
}

// Boundary nodes of every active lattice of a batch that has a mask: entries {lattice, node}.
template <typename S>
__global__ void __launch_bounds__(kRedThreads)
    batch_boundary_kernel(const BatchLat* __restrict__ lats, const int2* __restrict__ entries,
                          int n, const int* __restrict__ active, int parity,
                          const long long* __restrict__ tptr, int tstep, int stochastic) {
  using R = typename Traits<S>::R;
  uint32_t seed = 0;
  if (stochastic) {
    const long long t = *tptr + tstep;
    seed = (uint32_t)(t * 0x9E3779B1ull) ^ (uint32_t)(t >> 32);
  }
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int2 e = entries[k];
    if (!active[e.x]) continue;
    const BatchLat* L = lats + e.x;
    const Co<R> c = make_co<R>(L->c);
    const S* src = static_cast<const S*>(L->buf[parity]);
    S* dst = static_cast<S*>(L->buf[parity ^ 1]);
    step_node<S, true>(L->g, c, src, dst, e.y, seed, stochastic);
  }
}

// Convergence measure of every active lattice in FP64: max over (T, ux, uy) of
// ||phi(t) - phi(t - K)||_2 / (K ||phi(t)||_2), against the snapshot taken at
// the previous check, which is then replaced.  Comparing states K (even) steps
// apart is blind to the period-2 oscillation a closed cavity can keep at a
// small amplitude, which would otherwise hold a one-step residual above the
// tolerance.  Two deterministic stages: block (i, ch) sums chunk ch
// (kResChunk nodes) of lattice i into part[i][ch][0..7]; one thread per
// lattice then adds its chunks in order.
constexpr int kResChunk = 8192;

template <typename S>
__global__ void __launch_bounds__(kRedThreads)
    batch_residual_partial_kernel(const BatchLat* __restrict__ lats, const int* __restrict__ active,
                                  double* __restrict__ part, int maxchunks) {
  const int i = blockIdx.x, ch = blockIdx.y;
  if (!active[i]) return;
  const BatchLat* L = lats + i;
  const DevGeom& g = L->g;
  const long long n = (long long)g.ny * g.nx;
  const long long k0 = (long long)ch * kResChunk;
  if (k0 >= n) return;
  const long long k1 = k0 + kResChunk < n ? k0 + kResChunk : n;
  const S* cur = static_cast<const S*>(L->buf[0]);
  double* snap = L->snap;
  // per-node values and per-thread sums (at most kResChunk / blockDim nodes)
  // in the collision's arithmetic (FP32 below FP64 storage, where FP64 is
  // slow); block sums in FP64
  using R = typename Traits<S>::R;
  const Co<R> co = make_co<R>(L->c);
  const bool vh = L->c.vh != 0;
  R a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
    const int y = (int)(k / g.nx), x = (int)(k - (long long)y * g.nx);
    const long long idx = (long long)y * g.pitch + x;
    if (g.flags && (g.flags[idx] & kFlagSolid)) continue;
    R r1, u1, v1, t1;
    node_macros_r(co, vh, cur, g.plane, idx, r1, u1, v1, t1);
    const R t0 = (R)snap[k], u0 = (R)snap[n + k], v0 = (R)snap[2 * n + k];
    a[0] += (t1 - t0) * (t1 - t0);
    a[1] += t1 * t1;
    a[2] += (u1 - u0) * (u1 - u0);
    a[3] += u1 * u1;
    a[4] += (v1 - v0) * (v1 - v0);
    a[5] += v1 * v1;
    if (!isfinite(r1) || !isfinite(u1) || !isfinite(v1) || !isfinite(t1)) a[6] += R(1);
    snap[k] = t1;
    snap[n + k] = u1;
    snap[2 * n + k] = v1;
  }
  double acc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = (double)a[q];
  __shared__ double tot[8];
  block_sum_store<8>(acc, tot);
  __syncthreads();
  if (threadIdx.x < 8) part[((long long)i * maxchunks + ch) * 8 + threadIdx.x] = tot[threadIdx.x];
}

template <typename S>
__global__ void batch_residual_final_kernel(const BatchLat* __restrict__ lats, const int* __restrict__ active,
                                            int* __restrict__ snap_valid, const double* __restrict__ part,
                                            int maxchunks, double* __restrict__ res, int n, int K) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || !active[i]) return;
  const DevGeom& g = lats[i].g;
  const long long nodes = (long long)g.ny * g.nx;
  const int nch = (int)((nodes + kResChunk - 1) / kResChunk);
  double tot[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int ch = 0; ch < nch; ++ch)
    for (int q = 0; q < 8; ++q) tot[q] += part[((long long)i * maxchunks + ch) * 8 + q];
  double best = 0.0;
  for (int q = 0; q < 3; ++q) {
    const double den = sqrt(tot[2 * q + 1]) > 1e-30 ? sqrt(tot[2 * q + 1]) : 1e-30;
    const double v = sqrt(tot[2 * q]) / den;
    best = v > best ? v : best;
  }
  best /= (double)K;
  if (!snap_valid[i]) best = 1e300;
  if (tot[6] != 0.0 || !isfinite(best)) best = INFINITY;
  res[i] = best;
  snap_valid[i] = 1;
}

// a <- (a + b) / 2 over every stored value (both post-collision states of a
// lattice, one step apart): cancels any component that flips sign each step.
template <typename S>
__global__ void average_state_kernel(S* __restrict__ a, const S* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    using R = typename Traits<S>::R;
    const R v = R(0.5) * (to_r(a[i]) + to_r(b[i]));
    a[i] = from_r<S, R>(v);
  }
}

}  // namespace clbm

#include "clbm_resident.cuh"

namespace clbm {

// ---------------------------------------------------------------------------
// Launchers for one storage type
// ---------------------------------------------------------------------------
template <typename S>
struct LaunchImpl {
  static constexpr int V = Traits<S>::V;

  template <int VV>
  static cudaError_t box_step(const StepArgs& a, cudaStream_t s) {
    const int tiles = (a.g.nx + 32 * VV - 1) / (32 * VV), rows = a.g.yhi - a.g.ylo;
    const int wx = std::min(tiles, kStepThreads / 32), xblocks = wx > 0 ? (tiles + wx - 1) / wx : 0;
    if (xblocks <= 0 || rows <= 0) return cudaSuccess;
    const unsigned nblk = (unsigned)xblocks * (unsigned)rows;
    return launch_step(a.c.vh ? step_box_kernel<S, VV, true> : step_box_kernel<S, VV, false>, nblk, 32 * wx, s, a,
                       xblocks, rows);
  }

  // a step's launch; of more than one wave it may begin while its predecessor in the stream runs
  template <class... P, class... A>
  static cudaError_t launch_step(void (*kernel)(P...), unsigned blocks, int threads, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = (long long)blocks > (long long)sm_count() * kStepBlocks<S> ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  }

  static int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
      sms = 152;
    return sms;
  }

  static cudaError_t step(const StepArgs& a, cudaStream_t s) {
    if (!a.g.flags && !a.g.moving) {
      // FP64: an FP64 instruction holds a warp's quarter of the multiprocessor for 64 cycles, so a
      // step is as long as the most nodes that one lane of a quarter updates; tiles of one node a
      // lane where that number is then smaller (48^2: 12.1 -> 9 us a step)
      if constexpr (sizeof(S) == 8) {
        const long long quarters = 4LL * sm_count(), rows = a.g.yhi - a.g.ylo;
        const long long w1 = rows * ((a.g.nx + 31) / 32), w2 = rows * ((a.g.nx + 63) / 64);
        if ((w1 + quarters - 1) / quarters < 2 * ((w2 + quarters - 1) / quarters)) return box_step<1>(a, s);
      }
      return box_step<V>(a, s);
    }
    const int tiles = (a.g.nx + 32 * V - 1) / (32 * V);  // of a row
    // interior tiles: the own rows that are not next to a box wall (those are
    // boundary rows, in the node list).  Fewer than 2^31 blocks: a lattice has
    // at most 2^31 nodes, and each block updates more than one.
    const int xblocks = (tiles + kStepThreads / 32 - 1) / (kStepThreads / 32);
    const int y0 = a.g.ylo + a.g.ywlo;
    const int rows = std::max(0, a.g.yhi - a.g.ywhi - y0);
    const int nbb = (a.nb + kStepThreads - 1) / kStepThreads;
    const unsigned nblk = (unsigned)nbb + (unsigned)xblocks * (unsigned)rows;
    if (nblk == 0) return cudaSuccess;
    auto kernel = a.g.flags ? (a.c.vh ? step_fused_kernel<S, true, true> : step_fused_kernel<S, false, true>)
                            : (a.c.vh ? step_fused_kernel<S, true, false> : step_fused_kernel<S, false, false>);
    return launch_step(kernel, nblk, kStepThreads, s, a, nbb, xblocks, y0, rows);
  }

  static int blocks_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 4096) b = 4096;
    if (b < 1) b = 1;
    return (int)b;
  }

  static cudaError_t init(const DevGeom& g, const DevCoef& c, void* dst, const double* rho,
                          const double* ux, const double* uy, const double* T, cudaStream_t s) {
    if (g.ny <= 0 || g.pitch <= 0) return cudaSuccess;
    const dim3 grid((g.pitch + 255) / 256, g.ny < 65535 ? g.ny : 65535);
    init_kernel<S><<<grid, 256, 0, s>>>(g, c, static_cast<S*>(dst), rho, ux, uy, T);
    return cudaGetLastError();
  }

  static cudaError_t moments(const DevGeom& g, const DevCoef& c, const void* buf, double* rho,
                             double* ux, double* uy, double* T, cudaStream_t s) {
    const int rows = g.yhi - g.ylo;
    if (rows <= 0 || g.nx <= 0) return cudaSuccess;
    const int threads = g.nx >= 256 ? 256 : (g.nx + 31) / 32 * 32;
    const dim3 grid((g.nx + threads - 1) / threads, rows < 65535 ? rows : 65535);
    moments_kernel<S><<<grid, threads, 0, s>>>(g, c, static_cast<const S*>(buf), rho, ux, uy, T);
    return cudaGetLastError();
  }

  static cudaError_t residual(const DevGeom& g, const DevCoef& c, const void* cur,
                              const void* prev, double* partials, int nblocks, cudaStream_t s) {
    residual_kernel<S><<<nblocks, kRedThreads, 0, s>>>(g, c, static_cast<const S*>(cur),
                                                        static_cast<const S*>(prev), partials);
    return cudaGetLastError();
  }

  static cudaError_t totals(const DevGeom& g, const void* buf, double* partials, int nblocks,
                            cudaStream_t s) {
    totals_kernel<S><<<nblocks, kRedThreads, 0, s>>>(g, static_cast<const S*>(buf), partials);
    return cudaGetLastError();
  }

  static cudaError_t nusselt(const DevGeom& g, const DevCoef& c, const void* buf,
                             const NuLink* links, int nlinks, double* partials, int nblocks,
                             cudaStream_t s) {
    nusselt_kernel<S><<<nblocks, kRedThreads, 0, s>>>(g, c, static_cast<const S*>(buf), links,
                                                       nlinks, partials);
    return cudaGetLastError();
  }

  // batches run without the viscous source (clbm_batch_create rejects it)
  template <int VV>
  static const void* batch_kernel(int masked) {
    return masked ? (const void*)batch_step_kernel<S, VV, true> : (const void*)batch_step_kernel<S, VV, false>;
  }
  static const void* batch_kernel_of(int v, int masked) {
    if (v == 1) return batch_kernel<1>(masked);
    if (v == 2) return batch_kernel<2>(masked);
    if constexpr (V >= 4) {
      if (v == 4) return batch_kernel<4>(masked);
    }
    return nullptr;
  }

  static cudaError_t batch_step(int v, int masked, const BatchLat* lats, const int4* tiles, const int* count,
                                int parity, const long long* t, int tstep, int stochastic, int grid,
                                cudaStream_t s) {
    const void* k = batch_kernel_of(v, masked);
    if (!k) return cudaErrorInvalidValue;
    void* args[] = {&lats, &tiles, &count, &parity, &t, &tstep, &stochastic};
    return cudaLaunchKernel(k, dim3(grid), dim3(kStepThreads), args, 0, s);
  }

  static cudaError_t batch_boundary(const BatchLat* lats, const int2* entries, int n,
                                    const int* active, int parity, const long long* t, int tstep,
                                    int stochastic, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    int blocks = (n + kRedThreads - 1) / kRedThreads;
    if (blocks > 4096) blocks = 4096;
    batch_boundary_kernel<S><<<blocks, kRedThreads, 0, s>>>(lats, entries, n, active, parity, t,
                                                             tstep, stochastic);
    return cudaGetLastError();
  }

  static int batch_grid(int v, int masked) {
    int per_sm = 0;
    const void* k = batch_kernel_of(v, masked);
    if (!k) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kStepThreads, 0) != cudaSuccess) return 0;
    return sm_count() * (per_sm > 0 ? per_sm : 1);
  }

  static cudaError_t batch_residual(const BatchLat* lats, const int* active, int* snap_valid,
                                    double* res, int n, int K, double* part, int maxchunks,
                                    cudaStream_t s) {
    batch_residual_partial_kernel<S><<<dim3(n, maxchunks), kRedThreads, 0, s>>>(lats, active, part,
                                                                                maxchunks);
    batch_residual_final_kernel<S><<<(n + 255) / 256, 256, 0, s>>>(lats, active, snap_valid, part,
                                                                 maxchunks, res, n, K);
    return cudaGetLastError();
  }

  static cudaError_t average(void* a, const void* b, long long n, cudaStream_t s) {
    average_state_kernel<S><<<blocks_for(n, 256), 256, 0, s>>>(static_cast<S*>(a),
                                                                 static_cast<const S*>(b), n);
    return cudaGetLastError();
  }

  static size_t resident_smem(int nx, int rows, int nb, int vh) {
    return resident_bytes<S>(nx, rows, nb, vh != 0);
  }


  static cudaLaunchConfig_t resident_config(int cl, int n, int threads, size_t smem, cudaStream_t s,
                                            cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cl * n));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)cl;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
  }

  // the kernel with the limits that its launches may need
  static cudaError_t resident_prepare(int vh) {
    auto k = vh ? resident_kernel<S, true> : resident_kernel<S, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxResidentSmem);
    return e ? e : cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }

  static int resident_clusters(int cl, int threads, size_t smem, int vh) {
    int n = 0;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = resident_config(cl, 1, threads, smem, nullptr, &attr);
    if (resident_prepare(vh) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, vh ? resident_kernel<S, true> : resident_kernel<S, false>, &cfg) !=
            cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return n;
  }

  static cudaError_t resident_step(const ResArgs& a, int n, int threads, size_t smem, int vh, cudaStream_t s) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = resident_config(a.cl, n, threads, smem, s, &attr);
    return cudaLaunchKernelEx(&cfg, vh ? resident_kernel<S, true> : resident_kernel<S, false>, a);
  }

  static Launchers table() {
    Launchers L;
    L.resident_smem = &resident_smem;
    L.resident_clusters = &resident_clusters;
    L.resident_step = &resident_step;
    L.average = &average;
    L.batch_step = &batch_step;
    L.batch_boundary = &batch_boundary;
    L.batch_grid = &batch_grid;
    L.batch_residual = &batch_residual;
    L.residual_chunk = kResChunk;
    L.vec = V;
    L.step = &step;
    L.init = &init;
    L.moments = &moments;
    L.residual = &residual;
    L.nusselt = &nusselt;
    L.totals = &totals;
    L.elem_bytes = sizeof(S);
    return L;
  }
};

}  // namespace clbm
