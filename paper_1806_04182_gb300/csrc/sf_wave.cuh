// Scalar wave equation, first-order form (Sec. IV.A): fields
// (phi, Pi, d_x, d_y, d_z) with d_i = partial_i phi,
//   d/dt phi = -Pi,  d/dt Pi = -sum_i D_i d_i,  d/dt d_i = -D_i Pi,
// plus Kreiss-Oliger dissipation on every field (Sec. II.B.1).  The adjoint
// variant applies the transpose on the periodic grid: D_i^T = -D_i,
// Q_d^T = Q_d, so d/dt l_phi = Q l_phi, d/dt l_Pi = -l_phi + sum_i D_i l_d_i,
// d/dt l_d_i = D_i l_Pi.
#pragma once
#include "sf_common.cuh"

namespace sf {

// Right-hand side of one point: `ld(f, d, o)` reads field f at offset o along
// direction d, v[f] are the centre values.
//
// double: per field and direction the KO sum takes three pair sums and three
// fused multiply-adds with the weights of PatchArgs::cst, the centre one
// product per field, and a derivative two differences and two fused
// multiply-adds into the equation it enters: 121 operations a point (139 with
// the stencils evaluated apart), which the FP64 kernel's time follows (64^3
// stage 80 -> 74 us).  float is bound by its reads and keeps the stencils apart.
template <typename T, bool ADJ, typename Ld>
__device__ __forceinline__ void wave_rhs(const PatchArgs<T>& a, Ld&& ld, const T v[5], T r[5]) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int f = 0; f < 5; ++f) r[f] = a.cst[5].v[3] * v[f];
    r[ADJ ? 1 : 0] -= v[ADJ ? 0 : 1];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T k1 = a.cst[3].v[d], k2 = a.cst[4].v[d], k3 = a.cst[2].v[d];
      const T c1 = ADJ ? a.cst[1].v[d] : -a.cst[1].v[d], c2 = ADJ ? a.cst[0].v[d] : -a.cst[0].v[d];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        const T m1 = ld(f, d, -1), p1 = ld(f, d, 1), m2 = ld(f, d, -2), p2 = ld(f, d, 2);
        const T m3 = ld(f, d, -3), p3 = ld(f, d, 3);
        r[f] = fma(k1, m1 + p1, fma(k2, m2 + p2, fma(k3, m3 + p3, r[f])));
        // D_d Pi enters d_d's equation, D_d d_d that of Pi (with the sign -1, adjoint +1)
        if (f == 1) r[2 + d] = fma(c1, p1 - m1, fma(c2, m2 - p2, r[2 + d]));
        if (f == 2 + d) r[1] = fma(c1, p1 - m1, fma(c2, m2 - p2, r[1]));
      }
    }
  } else {
    auto D = [&](int f, int d) {
      return ((ld(f, d, -2) - ld(f, d, 2)) + T(8) * (ld(f, d, 1) - ld(f, d, -1))) * a.i12h[d];
    };
    auto delta6 = [&](int f, int d) {
      return (ld(f, d, -3) + ld(f, d, 3)) - T(6) * (ld(f, d, -2) + ld(f, d, 2)) +
             T(15) * (ld(f, d, -1) + ld(f, d, 1)) - T(20) * v[f];
    };
    const T div = D(2, 0) + D(3, 1) + D(4, 2);
    if (!ADJ) {
      r[0] = -v[1];
      r[1] = -div;
#pragma unroll
      for (int d = 0; d < 3; ++d) r[2 + d] = -D(1, d);
    } else {
      r[0] = T(0);
      r[1] = div - v[0];
#pragma unroll
      for (int d = 0; d < 3; ++d) r[2 + d] = D(1, d);
    }
#pragma unroll
    for (int f = 0; f < 5; ++f)
      r[f] += a.ko[0] * delta6(f, 0) + a.ko[1] * delta6(f, 1) + a.ko[2] * delta6(f, 2);
  }
}

// The same with every read from global memory (u: the point in field 0).
template <typename T, bool ADJ>
__device__ __forceinline__ void wave_point(const PatchArgs<T>& a, const T* u, T v[5],
                                           T r[5]) {
#pragma unroll
  for (int f = 0; f < 5; ++f) v[f] = u[f * a.sf];
  wave_rhs<T, ADJ>(
      a,
      [&](int f, int d, int o) {
        return u[f * a.sf + o * (d == 0 ? 1LL : (d == 1 ? a.sy : a.sz))];
      },
      v, r);
}

// The RK stage of one point.
template <typename T, bool ADJ>
__device__ __forceinline__ void wave_stage_point(const PatchArgs<T>& a, const StageArgs& s, int i, int j,
                                                 int k) {
  const int g = a.g;
  const long long c = (long long)(k + g) * a.sz + (long long)(j + g) * a.sy + (i + g);
  T v[5], r[5];
  // The RK inputs are read first, beside the stencils: read field by field in
  // the stage write, behind the stores of the field before, they made five
  // round trips to memory one after another (a 16^3 stage is nothing but
  // latency: 8.2 us, then 6.2; the bound on registers lets the compiler keep
  // more loads in flight).
  T un[5], acc[5], kh[5];
  const bool rk4 = s.rk == SF_RK4;
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const long long o = f * a.sf + c;
    un[f] = s.un_alias ? T(0) : a.un[o];
    acc[f] = (rk4 && s.stage > 0) ? a.acc[o] : T(0);
    kh[f] = (rk4 && s.stage == 3 && s.kahan) ? a.kh[o] : T(0);
  }
  wave_point<T, ADJ>(a, a.us + c, v, r);
  const Images im = ghost_images(a, s, i, j, k);
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const long long o = f * a.sf + c;
    r[f] = stage_combine(a, s, o, v[f], un[f], acc[f], kh[f], r[f]);
    a.nx[o] = r[f];
    if (s.check_finite && !finite_(r[f])) atomicOr(s.status, ST_NONFINITE);
  }
  if (im.mask) {
#pragma unroll
    for (int f = 0; f < 5; ++f) store_images(a, im, f * a.sf + c, r[f]);
  }
}

}  // namespace sf
