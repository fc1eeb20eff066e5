// Per-face arithmetic of the MHD stage kernel on pairs of values: the WENO
// reconstruction (App. A, App. B) of both edges of a cell for two fields at
// once, and the local Lax-Friedrichs flux (Eq. LLF) with the left and right
// states of a face as the two lanes.  For float a pair is an F2, each step
// one f32x2 instruction; for double it is two scalars.
//
// Both edges of a cell share everything but their linear weights: with the
// differences d_k = w_{k+1} - w_k, the candidate polynomials at the right edge
// are w_2 + (4 d_2 - d_3)/6, w_2 + (d_1 + 2 d_2)/6 and w_2 + (5 d_1 - 2 d_0)/6, at
// the left edge the mirror images, and the nonlinear weights are linear weight
// x P_k with the same P_k for both edges.  The edge value is the cell's value
// plus the weighted corrections, so a uniform state is reproduced exactly.
// Each correction holds only differences of its own stencil: a jump enters
// through the stencils that its weights switch off and nowhere else.  (With
// d_2/2 taken out of the three, two operations fewer, a jump J beside the cell
// had to cancel against it and left an error of eps J: float edge values wrong
// by 14% beside a jump by 10^6, now by 1e-7.)  43 operations give both edges
// (double) (App. B evaluated per face and per side takes about 124 for the
// same two values).
#pragma once

#include "sf_f2.cuh"
#include "sf_internal.cuh"

namespace sf {

template <typename T>
struct MhdCoef {
  T gamma;
  T eps[3];   // WENO epsilon per direction
  T q;        // WENO-Z exponent
  int variant;
  int split;  // 1: reconstruction of the Lax-Friedrichs split fluxes
  T idx[3];   // 1/dx_d
};

template <typename T>
__device__ __forceinline__ T wz_pow(T x, T q) {
  return q == T(2) ? x * x : (q == T(1) ? x : pow(x, q));
}

// ------------------------------------------------------------ pairs
// Two doubles; the compiler contracts none of these (explicit rounding), so
// every copy of the face code rounds alike.
struct R2 {
  double x, y;
  R2() = default;
  __device__ __forceinline__ R2(double a, double b) : x(a), y(b) {}
  __device__ __forceinline__ explicit R2(double v) : x(v), y(v) {}
};
__device__ __forceinline__ R2 add2(R2 a, R2 b) { return R2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)); }
__device__ __forceinline__ R2 sub2(R2 a, R2 b) { return R2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y)); }
__device__ __forceinline__ R2 mul2(R2 a, R2 b) { return R2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)); }
__device__ __forceinline__ R2 fma2(R2 a, R2 b, R2 c) {
  return R2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ R2 neg2(R2 a) { return R2(-a.x, -a.y); }

template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
  using type = F2;
};
template <>
struct PairOf<double> {
  using type = R2;
};

// -1/x.  float: the hardware approximation and one Newton step; double: the
// approximation rcp.approx.ftz.f64 (relative error below 2^-20) and one step
// of Householder's cubic iteration z (1 + e + e^2), e = 1 + x z (error below
// 2^-60 before rounding): 3 FP64 operations where the IEEE quotient takes
// about 9, on a pipe that issues one warp instruction every 16 cycles per SM.
// Exponents at which the approximation flushes or overflows take the IEEE
// division.  (The negative, because f32x2 has no negated operands: the sign
// goes into the scalar approximation for free.)
__device__ __forceinline__ float nrecip_approx(float x) {
  float z;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(-x));
  return z;
}
__device__ __forceinline__ F2 nrecip2(F2 x) {
  const F2 z(nrecip_approx(x.x), nrecip_approx(x.y));
  return fma2(z, fma2(x, z, F2(1.0f)), z);
}
// HALF: -1/(2x), the half by one off the approximation's exponent
template <bool HALF>
__device__ __forceinline__ double nrecip1(double x) {
  const unsigned ex = (unsigned)__double2hiint(x) & 0x7ff00000u;
  if (ex - 0x00400000u >= 0x7f800000u - 0x00400000u) return (HALF ? -0.5 : -1.0) / x;
  double z;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(-x));
  const double e = __fma_rn(x, z, 1.0);
  if (HALF) z = __hiloint2double(__double2hiint(z) - 0x00100000, __double2loint(z));
  return __fma_rn(z, __fma_rn(e, e, e), z);
}
__device__ __forceinline__ R2 nrecip2(R2 x) { return R2(nrecip1<false>(x.x), nrecip1<false>(x.y)); }

// Square root, 0 of a negative value (of a rounding error: the discriminant's,
// or that of the sum under the root of the signal speed of a state with
// negative pressure); NaN stays.  float: h = x rsqrt(x) and one Newton step h
// (3/2 - h rsqrt(x) / 2), x no less than 1e-37.
__device__ __forceinline__ F2 root2(F2 x) {
  auto up = [](float v) {
    float r;
    asm("max.NaN.f32 %0, %1, 0f02081CEA;" : "=f"(r) : "f"(v));  // 1e-37
    return r;
  };
  auto rs = [](float v) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
  };
  x = F2(up(x.x), up(x.y));
  const F2 y(rs(x.x), rs(x.y));
  const F2 h = mul2(x, y);
  return fma2(h, fma2(mul2(y, F2(-0.5f)), h, F2(0.5f)), h);
}
// double: h = x y with y = rsqrt.approx.ftz.f64, e = 1 - h y, and Halley's
// cubic step h (1 + e/2 + 3 e^2/8): 5 FP64 operations; exponents near the ends
// of the range (zero, inf and NaN among them) take the IEEE root.
__device__ __forceinline__ double sqrt1(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  if (hi - 0x00400000u >= 0x7f800000u - 0x00400000u) return sqrt(x);  // a set sign bit too
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = __dmul_rn(x, y), e = __fma_rn(-h, y, 1.0);
  return __fma_rn(__dmul_rn(h, e), __fma_rn(0.375, e, 0.5), h);
}
__device__ __forceinline__ double nonneg(double x) {  // by the sign bit, off the FP64 pipe
  return (unsigned)__double2hiint(x) - 0x80000000u < 0x7ff00000u ? 0.0 : x;  // finite, < 0
}
__device__ __forceinline__ R2 root2(R2 x) { return R2(sqrt1(nonneg(x.x)), sqrt1(nonneg(x.y))); }

__device__ __forceinline__ F2 abs2(F2 x) { return F2(fabsf(x.x), fabsf(x.y)); }
__device__ __forceinline__ R2 abs2(R2 x) { return R2(fabs(x.x), fabs(x.y)); }
// the larger of two non-negative values; double: as integers (their bits are
// ordered alike)
__device__ __forceinline__ float larger(float a, float b) { return a > b ? a : b; }
__device__ __forceinline__ double larger(double a, double b) {
  return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}

// ------------------------------------------------------------ reconstruction
// 2^-floor(log2 m) of a normal m < 2^127
__device__ __forceinline__ float inv_pow2(float m) {
  return __int_as_float(0x7f000000 - (__float_as_int(m) & 0x7f800000));
}

// Nonlinear weights P_k (without their linear weights) from E_k = eps + beta_k,
// up to a common factor.
//
// JS weights are 1/E_k^2; over the common denominator P_0 = (E_1 E_2)^2 and
// so on, one division fewer.  In float the products E_i E_j are scaled by the
// power of two of the largest first, so that the largest P_k lies in [1, 4)
// whatever the units.  Where a product leaves the range of that scale (E_k
// above 9e18: jumps of 3e9) P_k = (E_min / E_k)^2, in [0, 1], the largest 1; a
// weight below the range of a float is nil, as 1/E_k^2 is.  (128^3 step 919 us;
// without that form 911, with it for all cells 931, the test shared by two or
// four pairs of fields, whose values then wait for it in registers, 960 and
// 1056.)
template <int VAR>
__device__ __forceinline__ void weno_weights(F2 e0, F2 e1, F2 e2, const MhdCoef<float>& mc, F2& p0,
                                             F2& p1, F2& p2) {
  if constexpr (VAR == 1) {
    // 1 + (tau / E_k)^q, times the q-th power of a scale u: beyond ratios of
    // 2^30 (a jump of 2 beside a uniform state on 128 cells) the inverse power
    // of two of the largest, so that the weights and their sums stay in range.
    // q = 2 in a branch of its own for all of it (64^3 step 354 -> 247 us; 318
    // without the scale and with the power chosen value by value)
    const F2 tau = abs2(sub2(e0, e2));
    auto ratio = [&](F2 e) { return F2(fminf(tau.x / e.x, 1.5e38f), fminf(tau.y / e.y, 1.5e38f)); };
    F2 r0 = ratio(e0), r1 = ratio(e1), r2 = ratio(e2);
    auto scale = [](float a, float b, float c) {
      const float m = fmaxf(fmaxf(a, b), c);
      return m < 0x1p30f ? 1.0f : inv_pow2(m);
    };
    const F2 u(scale(r0.x, r1.x, r2.x), scale(r0.y, r1.y, r2.y));
    r0 = mul2(r0, u);
    r1 = mul2(r1, u);
    r2 = mul2(r2, u);
    if (mc.q == 2.0f) {
      const F2 one = mul2(u, u);
      p0 = fma2(r0, r0, one);
      p1 = fma2(r1, r1, one);
      p2 = fma2(r2, r2, one);
    } else {
      auto power = [&](F2 r) { return F2(wz_pow(r.x, mc.q), wz_pow(r.y, mc.q)); };
      const F2 one = power(u);
      p0 = add2(one, power(r0));
      p1 = add2(one, power(r1));
      p2 = add2(one, power(r2));
    }
  } else {
    p0 = mul2(e1, e2);
    p1 = mul2(e0, e2);
    p2 = mul2(e0, e1);
    auto max3 = [](float a, float b, float c) { return fmaxf(fmaxf(a, b), c); };
    const float mx = max3(p0.x, p1.x, p2.x), my = max3(p0.y, p1.y, p2.y);
    if (fmaxf(mx, my) < 0x1p126f) {
      const F2 sc(inv_pow2(mx), inv_pow2(my));
      p0 = mul2(p0, sc);
      p1 = mul2(p1, sc);
      p2 = mul2(p2, sc);
    } else {
      const float lx = fminf(fminf(e0.x, e1.x), e2.x), ly = fminf(fminf(e0.y, e1.y), e2.y);
      auto w = [&](F2 e) {
        const F2 z = nrecip2(e);  // (E_k infinite: NaN, which the saturation takes to 0)
        return F2(__saturatef(-lx * z.x), __saturatef(-ly * z.y));
      };
      p0 = w(e0);
      p1 = w(e1);
      p2 = w(e2);
    }
    p0 = mul2(p0, p0);
    p1 = mul2(p1, p1);
    p2 = mul2(p2, p2);
  }
}
template <int VAR>
__device__ __forceinline__ void weno_weights(R2 e0, R2 e1, R2 e2, const MhdCoef<double>& mc, R2& p0,
                                             R2& p1, R2& p2) {
  if constexpr (VAR == 1) {
    const R2 tau = abs2(sub2(e0, e2));
    if (mc.q == 2.0) {  // (E_k^2 + tau^2) (E_i E_j)^2
      const R2 t2 = mul2(tau, tau);
      const R2 q0 = mul2(e0, e0), q1 = mul2(e1, e1), q2 = mul2(e2, e2);
      p0 = mul2(add2(q0, t2), mul2(q1, q2));
      p1 = mul2(add2(q1, t2), mul2(q0, q2));
      p2 = mul2(add2(q2, t2), mul2(q0, q1));
    } else {
      auto w = [&](R2 e) {
        return R2(1.0 + wz_pow(tau.x / e.x, mc.q), 1.0 + wz_pow(tau.y / e.y, mc.q));
      };
      p0 = w(e0);
      p1 = w(e1);
      p2 = w(e2);
    }
  } else {
    p0 = mul2(e1, e2);
    p1 = mul2(e0, e2);
    p2 = mul2(e0, e1);
    p0 = mul2(p0, p0);
    p1 = mul2(p1, p1);
    p2 = mul2(p2, p2);
  }
}

// -1/2 x the reciprocals of both sums.  float JS: the sums lie in [1, 64), so
// one reciprocal of their product serves both.
template <int VAR>
__device__ __forceinline__ void half_recips(F2 sr, F2 sl, F2& ir, F2& il) {
  if constexpr (VAR == 0) {
    const F2 h = mul2(nrecip2(mul2(sr, sl)), F2(0.5f));
    ir = mul2(h, sl);
    il = mul2(h, sr);
  } else {
    ir = mul2(nrecip2(sr), F2(0.5f));
    il = mul2(nrecip2(sl), F2(0.5f));
  }
}
template <int VAR>
__device__ __forceinline__ void half_recips(R2 sr, R2 sl, R2& ir, R2& il) {
  ir = R2(nrecip1<true>(sr.x), nrecip1<true>(sr.y));
  il = R2(nrecip1<true>(sl.x), nrecip1<true>(sl.y));
}

// Both edge values of cell c of two fields from w[0..4] = U_{c-2..c+2}: er,
// the left state at c + 1/2, and el, the right state at c - 1/2.  VAR 0
// WENO5-JS, 1 WENO5-Z, 2 WENO3.
template <int VAR, typename T, typename P>
__device__ __forceinline__ void weno_edges(const P* w, T eps, const MhdCoef<T>& mc, P& er, P& el) {
  const P d1 = sub2(w[2], w[1]), d2 = sub2(w[3], w[2]);
  if constexpr (VAR == 2) {
    const P ep(eps);
    P e0 = fma2(d2, d2, ep), e1 = fma2(d1, d1, ep);
    if constexpr (sizeof(T) == 4) {
      // scaled so that the larger one lies in [1, 2): the squares and their
      // products with the differences stay in range (capped: 1.5e38 < 2^127)
      auto cap = [](P e) { return P(fminf(e.x, 1.5e38f), fminf(e.y, 1.5e38f)); };
      e0 = cap(e0);
      e1 = cap(e1);
      const P sc(inv_pow2(fmaxf(e0.x, e1.x)), inv_pow2(fmaxf(e0.y, e1.y)));
      e0 = mul2(e0, sc);
      e1 = mul2(e1, sc);
    }
    const P p0 = mul2(e1, e1), p1 = mul2(e0, e0);
    // er = w_2 + (2 p0 d2 + p1 d1) / (2 (2 p0 + p1)), el its mirror image
    const P q0 = mul2(p0, d2), q1 = mul2(p1, d1), two(T(2));
    P ir, il;
    half_recips<VAR>(fma2(two, p0, p1), fma2(two, p1, p0), ir, il);
    er = fma2(fma2(P(T(-2)), q0, neg2(q1)), ir, w[2]);
    el = fma2(fma2(two, q1, q0), il, w[2]);
    return;
  }
  // beta_k = a_k (4/3 a_k -+ d) + d^2 (13/12 a^2 + 1/4 b^2 of App. B with b
  // expressed by a and a difference), d^2 + eps shared
  const P d0 = sub2(w[1], w[0]), d3 = sub2(w[4], w[3]);
  const P a0 = sub2(d3, d2), a1 = sub2(d2, d1), a2 = sub2(d1, d0);
  const P c43(T(4.0 / 3.0)), ep(eps);
  const P g1 = fma2(d1, d1, ep), g2 = fma2(d2, d2, ep);
  const P e0 = fma2(a0, fma2(c43, a0, neg2(d2)), g2);
  const P e1 = fma2(a1, fma2(c43, a1, d1), g1);
  const P e2 = fma2(a2, fma2(c43, a2, d1), g1);
  P p0, p1, p2;
  weno_weights<VAR>(e0, e1, e2, mc, p0, p1, p2);
  // right edge: weights 3 p0, 6 p1, p2; left edge: p0, 6 p1, 3 p2.  The weighted
  // corrections x 6 (left edge with opposite sign), 4 d_2 - d_3 = 3 d_2 - a_0 and
  // so on, grouped by difference: a factor of d_k or a_k holds the weights of
  // the stencils that contain it and no others
  const P two(T(2)), three(T(3)), ct(T(2.0 / 3.0));
  const P p01 = fma2(two, p1, p0), p12 = fma2(two, p1, p2);
  const P sr = fma2(three, p01, p2), sl = fma2(three, p12, p0);
  const P qa = mul2(p0, a0), qc = mul2(p2, a2);
  const P nr = fma2(d2, fma2(two, p01, p0), fma2(d1, p12, fma2(ct, qc, neg2(qa))));
  const P nl = fma2(d1, fma2(two, p12, p2), fma2(d2, p01, fma2(neg2(ct), qa, qc)));
  P ir, il;
  half_recips<VAR>(sr, sl, ir, il);
  er = fma2(neg2(nr), ir, w[2]);
  el = fma2(nl, il, w[2]);
}

// ------------------------------------------------------------ flux
// Twice the LLF flux through a face along D, FL + FR - S (UR - UL), from the
// states q[f] = (left, right).  Velocities and fluxes are carried negated
// (n...), see nrecip2.
template <int D, typename T, typename P>
__device__ __forceinline__ void llf_flux2(const P* q, T gamma, T* F) {
  constexpr int A = (D + 1) % 3, B = (D + 2) % 3;  // the other two directions
  const P nir = nrecip2(q[0]);
  const P nv[3] = {mul2(q[1], nir), mul2(q[2], nir), mul2(q[3], nir)};
  const P* b = q + 5;
  const P bd2 = mul2(b[D], b[D]);
  const P B2 = fma2(b[B], b[B], fma2(b[A], b[A], bd2));
  const P nSvB = fma2(q[3], nv[2], fma2(q[2], nv[1], fma2(q[1], nv[0], neg2(B2))));
  const P pr = mul2(P(gamma - T(1)), fma2(P(T(0.5)), nSvB, q[4]));
  const P pt = fma2(P(T(0.5)), B2, pr);
  const P nvB = fma2(nv[2], b[2], fma2(nv[1], b[1], mul2(nv[0], b[0])));
  const P nb = neg2(b[D]);
  const P Sd = q[1 + D];
  // signal speed |v_d| + c_fast
  const P na2 = mul2(mul2(P(gamma), pr), nir);
  const P h = mul2(P(T(-0.5)), fma2(B2, nir, na2));
  const P disc = fma2(neg2(na2), mul2(bd2, nir), mul2(h, h));
  const P cf = root2(add2(root2(disc), h));
  const T S = larger(fabs(nv[D].x) + cf.x, fabs(nv[D].y) + cf.y);
  auto out = [&](int f, P nf) { F[f] = fma(-S, q[f].y - q[f].x, -nf.x - nf.y); };
  F[0] = fma(-S, q[0].y - q[0].x, Sd.x + Sd.y);
  out(1 + D, sub2(fma2(Sd, nv[D], bd2), pt));
  // u v + w z of both states: in double one chain over the states
  auto out4 = [&](int f, P u, P v, P w, P z) {
    if constexpr (sizeof(T) == 8) {
      const T t = fma(w.y, z.y, fma(w.x, z.x, fma(u.y, v.y, u.x * v.x)));
      F[f] = fma(-S, q[f].y - q[f].x, -t);
    } else {
      out(f, fma2(w, z, mul2(u, v)));
    }
  };
  out4(1 + A, Sd, nv[A], b[D], b[A]);
  out4(1 + B, Sd, nv[B], b[D], b[B]);
  out4(4, add2(q[4], pt), nv[D], nb, nvB);
  F[5 + D] = fma(-S, b[D].y - b[D].x, T(0));
  out4(5 + A, nv[D], b[A], nb, nv[A]);
  out4(5 + B, nv[D], b[B], nb, nv[B]);
}

}  // namespace sf
