// CCZ4 right-hand side at one point in FP64: the equations of z4_rhs
// (sf_z4.cuh) in the fewest FP64 operations.
//
// The FP64 pipe takes one warp instruction per 16 cycles and SM and bounds
// every FP64 CCZ4 stage, so operations are what a point costs (with the stage
// write 2820 a point in z4_rhs's form, 2435 here).  z4_rhs keeps its order of
// operations, which fixes the bits of the float kernels; here
//  - stencil weights (PatchArgs::cst) folded into the sums (for the fields that
//    are 1 in flat space only as far as flat space stays exactly flat),
//    advection and KO in one accumulator, advection of the fields whose
//    derivatives serve nothing else (A~, B) straight from their differences;
//  - gt^{mn} d_m d_n of the metric as one weighted sum over its stencil, the
//    weights shared by the six components;
//  - contractions factored (gt^{ab} d_b chi, gt_ab (Gammahat - Gamma~)^b and the
//    covector of the A~ and gt^{ab} terms of d/dt Gammahat once each), diagonal
//    components of symmetrised products once and doubled, equal coefficients of
//    gt_ab and A~_ab added up first;
//  - reciprocals and the logarithm near 1 without IEEE's last half-bit
//    (recip64, ln64).
#pragma once
#include "sf_common.cuh"

namespace sf {

// 1/x: the hardware approximation rcp.approx.ftz.f64 (relative error below
// 2^-20) and one step of Householder's cubic iteration z (1 + e + e^2), e = 1 -
// x z: 3 operations where the IEEE quotient takes about 9.  Exponents at which
// the approximation flushes or overflows take the IEEE quotient.
__device__ __forceinline__ double recip64(double x) {
  const unsigned ex = (unsigned)__double2hiint(x) & 0x7ff00000u;
  if (ex - 0x00400000u >= 0x7f800000u - 0x00400000u) return 1.0 / x;
  double z;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(z) : "d"(x));
  const double e = fma(-x, z, 1.0);
  return fma(z, fma(e, e, e), z);
}
// ln d.  Near 1, where a conformal determinant stays, 2 atanh(z) with
// z = (d - 1)/(d + 1) by its series to z^13 (|z| < 1/32: the next term is below
// 2^-70 z); elsewhere log().
__device__ __forceinline__ double ln64(double d) {
  if (fabs(d - 1.0) >= 0.0625) return log(d);  // (NaN takes the series and stays NaN)
  const double z = (d - 1.0) * recip64(d + 1.0), y = z * z;
  double p = fma(y, 2.0 / 13.0, 2.0 / 11.0);
  p = fma(y, p, 2.0 / 9.0);
  p = fma(y, p, 2.0 / 7.0);
  p = fma(y, p, 2.0 / 5.0);
  p = fma(y, p, 2.0 / 3.0);
  return fma(y * z, p, z + z);
}

// What a field's cross is read for: advection and KO only; D_i; D_i and D_ii;
// D_i and the weighted sum of D_ii.
enum Z4Cross { Z4_ADV, Z4_DERIV, Z4_HESS, Z4_TRACE };

template <bool LOP, typename Src>
struct Z4Sten64 {
  const PatchArgs<double>& a;
  Src& src;
  double be[3];  // shift at the point
  double bh[3];  // be_d / (12 dx_d)
  // weights of the metric's trace: the second differences' per direction
  // (gt^dd / (12 dx_d^2)), the mixed ones' (2 gt^mn / (144 dx dx))
  double wd[3], wm[3];

  // cross of field f: returns beta^k d_k U + the KO term.  `one`: the field is
  // 1 in flat space, where small whole weights cancel exactly and folded ones
  // need not
  template <Z4Cross K>
  __device__ __forceinline__ double cross(int f, double* d, double* dd, bool one = false) {
    const long long st[3] = {1, src.sy(), src.sz()};
    const double* p = src.p(f);
    const double c = src.ld(p);
    double acc = one ? 0.0 : c * a.cst[5].v[3];
    if (K == Z4_TRACE) *dd = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const long long s = st[q];
      const double m1 = src.ld(p - s), p1 = src.ld(p + s);
      const double m2 = src.ld(p - 2 * s), p2 = src.ld(p + 2 * s);
      const double m3 = src.ld(p - 3 * s), p3 = src.ld(p + 3 * s);
      const double s1 = m1 + p1, s2 = m2 + p2, s3 = m3 + p3;
      if (one) {
        acc = fma(a.cst[2].v[q], fma(-20.0, c, fma(15.0, s1, fma(-6.0, s2, s3))), acc);
      } else {
        acc = fma(s1, a.cst[3].v[q], acc);
        acc = fma(s2, a.cst[4].v[q], acc);
        acc = fma(s3, a.cst[2].v[q], acc);
      }
      const double e = fma(8.0, p1 - m1, m2 - p2);  // 12 dx D
      if (K != Z4_ADV) d[q] = e * a.i12h[q];
      if (LOP) {
        // one-sided on the side the characteristic comes from (Sec. II.B.1)
        double ad = e;
        if (be[q] != 0.0)
          ad = be[q] > 0.0 ? (p3 - 6.0 * p2 + 18.0 * p1 - 10.0 * c - 3.0 * m1)
                           : (-m3 + 6.0 * m2 - 18.0 * m1 + 10.0 * c + 3.0 * p1);
        acc = fma(bh[q], ad, acc);
      } else if (K == Z4_ADV) {
        acc = fma(bh[q], e, acc);
      } else {
        acc = fma(be[q], d[q], acc);
      }
      const double e2 = fma(-30.0, c, fma(16.0, s1, -s2));  // 12 dx^2 D_dd
      if (K == Z4_HESS) dd[q] = e2 * a.i12h2[q];
      if (K == Z4_TRACE) *dd = fma(wd[q], e2, *dd);
    }
    return acc;
  }
  // 144 dx_m dx_n D_n(D_m) of field f
  __device__ __forceinline__ double mix(int f, int m, int n) const {
    const double* p = src.p(f);
    const long long st[3] = {1, src.sy(), src.sz()};
    const long long sa = st[m], sb = st[n];
    auto row = [&](long long o) {
      const double* q = p + o;
      return fma(8.0, src.ld(q + sa) - src.ld(q - sa), src.ld(q - 2 * sa) - src.ld(q + 2 * sa));
    };
    return fma(8.0, row(sb) - row(-sb), row(-2 * sb) - row(2 * sb));
  }
  // Hessian xx, xy, xz, yy, yz, zz and D_i of field f; returns advection + KO
  __device__ __forceinline__ double hess(int f, double* d, double* h, bool one = false) {
    double dd[3];
    const double acc = cross<Z4_HESS>(f, d, dd, one);
    h[0] = dd[0];
    h[3] = dd[1];
    h[5] = dd[2];
    h[1] = mix(f, 0, 1) * a.i144hh[0];
    h[2] = mix(f, 0, 2) * a.i144hh[1];
    h[4] = mix(f, 1, 2) * a.i144hh[2];
    return acc;
  }
  // D_i and gt^{mn} d_m d_n of field f; returns advection + KO
  __device__ __forceinline__ double trace(int f, double* d, double& t, bool one) {
    const double acc = cross<Z4_TRACE>(f, d, &t, one);
    t = fma(wm[0], mix(f, 0, 1), t);
    t = fma(wm[1], mix(f, 0, 2), t);
    t = fma(wm[2], mix(f, 1, 2), t);
    return acc;
  }
};

template <bool LOP, typename Src, typename Out>
__device__ __forceinline__ void z4_rhs64(const PatchArgs<double>& a, const Z4Coef<double>& zc, Src& src,
                                         Out&& out) {
  Z4Sten64<LOP, Src> sten{a, src};
  const double chi = src.centre(0), Kh = src.centre(7), Th = src.centre(17), al = src.centre(18);
  double gt[6], At[6], Gh[3];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    gt[q] = src.centre(1 + q);
    At[q] = src.centre(8 + q);
  }
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    sten.be[p] = src.centre(19 + p);
    sten.bh[p] = sten.be[p] * a.i12h[p];
    Gh[p] = src.centre(14 + p);
  }
  const double kz = zc.kappa_z;

  // ---- determinant, inverse and ln det of the conformal metric
  double ig[6], kcl;
  {
    const double c00 = fma(gt[3], gt[5], -gt[4] * gt[4]);
    const double c01 = fma(gt[2], gt[4], -gt[5] * gt[1]);
    const double c02 = fma(gt[1], gt[4], -gt[3] * gt[2]);
    const double c11 = fma(gt[0], gt[5], -gt[2] * gt[2]);
    const double c12 = fma(gt[1], gt[2], -gt[0] * gt[4]);
    const double c22 = fma(gt[0], gt[3], -gt[1] * gt[1]);
    const double det = fma(c02, gt[2], fma(c01, gt[1], c00 * gt[0]));
    const double idet = recip64(det);
    ig[0] = c00 * idet;
    ig[1] = c01 * idet;
    ig[2] = c02 * idet;
    ig[3] = c11 * idet;
    ig[4] = c12 * idet;
    ig[5] = c22 * idet;
    kcl = zc.kappa_c * (1.0 / 3.0) * al;
    kcl *= ln64(det);  // kappa_c alpha ln(det) / 3
  }
  // gt^{ij} X_ij of a symmetric X stored as xx, xy, xz, yy, yz, zz
  auto trg = [&](const double* X) {
    const double dg = fma(ig[5], X[5], fma(ig[3], X[3], ig[0] * X[0]));
    return fma(2.0, fma(ig[4], X[4], fma(ig[2], X[2], ig[1] * X[1])), dg);
  };
  const double trA3 = trg(At) * (1.0 / 3.0);
  const double ichi = recip64(chi);
  const double Kt = fma(2.0, Th, Kh);

  // ---- shift: first derivatives, gt^{mn} d_m d_n beta^c and d_b d_k beta^k
  double dbe[3][3], betaAcc[3], rGh[3], sA[6], d23;  // d23: 2/3 div beta
  {
    double ddiv[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double h[6];
      betaAcc[c] = sten.hess(19 + c, dbe[c], h);
      rGh[c] = trg(h);
#pragma unroll
      for (int m = 0; m < 3; ++m) ddiv[m] += h[S(c, m)];
    }
    const double divbe = dbe[0][0] + dbe[1][1] + dbe[2][2];
    d23 = (2.0 / 3.0) * divbe;
#pragma unroll
    for (int m = 0; m < 3; ++m) ddiv[m] *= 1.0 / 3.0;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      double r = fma(Gh[p], d23, rGh[p]);
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        r = fma(-Gh[m], dbe[p][m], r);
        r = fma(ig[S(p, m)], ddiv[m], r);
      }
      rGh[p] = r;
    }
    // A~_pc d_b beta^c + A~_bc d_p beta^c
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        double t = At[S(p, 0)] * dbe[0][b];
        t = fma(At[S(p, 1)], dbe[1][b], t);
        t = fma(At[S(p, 2)], dbe[2][b], t);
        if (b == p) {
          t += t;
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) t = fma(At[S(c, b)], dbe[c][p], t);
        }
        sA[S(p, b)] = t;
      }
  }

  // ---- conformal metric: derivatives, d/dt gt (Eq. syseq1); Rt starts with
  // -1/2 gt^{mn} d_m d_n gt_q + 1/2 Gammahat^c d_c gt_q (the latter Gammahat^c
  // Gamma~_(pb)c)
  double Gl[3][6];  // Gamma~_{a bc}, first index lowered
  double Rt[6];
  {
    double dgt[6][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) sten.wd[d] = ig[S(d, d)] * a.i12h2[d];
    sten.wm[0] = (ig[1] + ig[1]) * a.i144hh[0];
    sten.wm[1] = (ig[2] + ig[2]) * a.i144hh[1];
    sten.wm[2] = (ig[4] + ig[4]) * a.i144hh[2];
    const double al2 = al + al;
    const double cg = fma(al2, trA3, -d23) - kcl;  // the coefficient of gt_q
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        const int q = S(p, b);
        double t1;
        double s = sten.trace(1 + q, dgt[q], t1, p == b);
        double t = gt[S(p, 0)] * dbe[0][b];
        t = fma(gt[S(p, 1)], dbe[1][b], t);
        t = fma(gt[S(p, 2)], dbe[2][b], t);
        if (b == p) {
          s = fma(2.0, t, s);
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) t = fma(gt[S(c, b)], dbe[c][p], t);
          s += t;
        }
        s = fma(-al2, At[q], s);
        out(1 + q, fma(cg, gt[q], s), gt[q]);
#pragma unroll
        for (int c = 0; c < 3; ++c) t1 = fma(-Gh[c], dgt[q][c], t1);
        Rt[q] = -0.5 * t1;
      }
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        // Gamma~_{p bb} and Gamma~_{p bc}, c the next direction
        const int c = (b + 1) % 3;
        Gl[p][S(b, b)] = p == b ? 0.5 * dgt[S(p, p)][p] : fma(-0.5, dgt[S(b, b)][p], dgt[S(p, b)][b]);
        if (p == b)
          Gl[p][S(b, c)] = 0.5 * dgt[S(p, p)][c];
        else if (p == c)
          Gl[p][S(b, c)] = 0.5 * dgt[S(p, p)][b];
        else
          Gl[p][S(b, c)] = 0.5 * (dgt[S(p, c)][b] + dgt[S(p, b)][c] - dgt[S(b, c)][p]);
      }
  }
  double Gu[3][6];  // Gamma~^a_{bc}
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 6; ++q)
      Gu[p][q] = fma(ig[S(p, 2)], Gl[2][q], fma(ig[S(p, 1)], Gl[1][q], ig[S(p, 0)] * Gl[0][q]));
  double y[3], yl[3];  // Gammahat^i - Gamma~^i = 2 Z^i / chi, and lowered
#pragma unroll
  for (int p = 0; p < 3; ++p) y[p] = Gh[p] - trg(Gu[p]);
  {
    const double k = -al * fma(2.0 / 3.0, Kt, kz);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      rGh[p] = fma(k, y[p], rGh[p]);
      yl[p] = fma(gt[S(p, 2)], y[2], fma(gt[S(p, 1)], y[1], gt[S(p, 0)] * y[0]));
    }
  }

  // ---- Gammahat: advection and KO of d/dt Gammahat, gt_c(p d_b) Gammahat^c into Rt
  double GhAK[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double d[3];
    GhAK[c] = sten.template cross<Z4_DERIV>(14 + c, d, nullptr);
    double hd[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) hd[b] = 0.5 * d[b];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        const int q = S(p, b);
        if (b == p) {
          Rt[q] = fma(gt[S(c, p)], d[p], Rt[q]);
        } else {
          Rt[q] = fma(gt[S(c, p)], hd[b], Rt[q]);
          Rt[q] = fma(gt[S(c, b)], hd[p], Rt[q]);
        }
      }
  }

  // ---- chi: derivatives; its right-hand side is complete here
  double dchi[3], ddchi[6];
  {
    const double r = sten.hess(0, dchi, ddchi, true);
    out(0, fma(chi, fma((2.0 / 3.0) * al, Kt, -d23), r), chi);
  }

  // ---- Ricci tensor Rhat_ab + Rchi_ab
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double Qc[3][3];  // gt^{nm} Gamma~^c_{mp}
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int n = 0; n < 3; ++n)
        Qc[p][n] = fma(ig[S(n, 2)], Gu[c][S(2, p)],
                       fma(ig[S(n, 1)], Gu[c][S(1, p)], ig[S(n, 0)] * Gu[c][S(0, p)]));
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        double s = Rt[S(p, b)];
        if (b == p) {
          double t = Qc[p][0] * Gl[p][S(c, 0)];
          t = fma(Qc[p][1], Gl[p][S(c, 1)], t);
          t = fma(Qc[p][2], Gl[p][S(c, 2)], t);
          s = fma(2.0, t, s);
#pragma unroll
          for (int n = 0; n < 3; ++n) s = fma(Qc[p][n], Gl[c][S(n, p)], s);
        } else {
#pragma unroll
          for (int n = 0; n < 3; ++n) {
            s = fma(Qc[p][n], Gl[b][S(c, n)], s);
            s = fma(Qc[p][n], Gl[c][S(n, b)], s);
            s = fma(Qc[b][n], Gl[p][S(c, n)], s);
          }
        }
        Rt[S(p, b)] = s;
      }
  }
  const double hichi = 0.5 * ichi;
  double uchi[3], w[3];  // gt^{ab} d_b chi; d_b chi / (2 chi)
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    uchi[p] = fma(ig[S(p, 2)], dchi[2], fma(ig[S(p, 1)], dchi[1], ig[S(p, 0)] * dchi[0]));
    w[p] = hichi * dchi[p];
  }
  {
    // Rchi = 1/(2 chi) (d d chi - Gamma~ d chi + v_p d_b chi + v_b d_p chi +
    // gt_pb tr), v_p = Z_p / (chi/2) - d_p chi / (4 chi)
    double v[3];
    double tr = trg(ddchi);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v[c] = fma(-0.5, w[c], yl[c]);
      tr = fma(-Gh[c], dchi[c], tr);
      tr = fma(-3.0 * w[c], uchi[c], tr);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        const int q = S(p, b);
        double X = fma(gt[q], tr, ddchi[q]);
        X = fma(-Gu[0][q], dchi[0], X);
        X = fma(-Gu[1][q], dchi[1], X);
        X = fma(-Gu[2][q], dchi[2], X);
        X = fma(v[p], dchi[b], X);
        X = fma(v[b], dchi[p], X);
        Rt[q] = fma(hichi, X, Rt[q]);
      }
  }
  const double trR = trg(Rt);

  // ---- alpha: derivatives; its right-hand side is complete here
  double dal[3], M[6], trD;  // M_ab = alpha R_ab - D_a D_b alpha
  {
    double h[6];
    const double r = sten.hess(18, dal, h, true);
    out(18, fma(zc.slicing == 0 ? -(al + al) : -al * al, Kh, r), al);
    double g2 = uchi[0] * dal[0];
    g2 = fma(uchi[1], dal[1], g2);
    g2 = fma(uchi[2], dal[2], g2);
    g2 *= -hichi;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        const int q = S(p, b);
        double X = fma(gt[q], g2, h[q]);
        X = fma(-Gu[0][q], dal[0], X);
        X = fma(-Gu[1][q], dal[1], X);
        X = fma(-Gu[2][q], dal[2], X);
        X = fma(dal[p], w[b], X);
        h[q] = fma(dal[b], w[p], X);
        M[q] = fma(al, Rt[q], -h[q]);
      }
    trD = trg(h);
  }

  // ---- A~ contractions; the terms of d/dt Gammahat with A~^{ab}; r0: d/dt A~
  // without advection and KO
  double r0[6], AA;
  {
    double Aud[3][3];  // A~^a_b = gt^{ac} A~_cb
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        Aud[p][b] = fma(ig[S(p, 2)], At[S(2, b)], fma(ig[S(p, 1)], At[S(1, b)], ig[S(p, 0)] * At[S(0, b)]));
    const double trM3 = fma(al, trR, -trD) * (1.0 / 3.0);
    const double cg = -fma(chi, trM3, zc.kappa_c * al * trA3);  // coefficients of gt_q, A~_q
    const double ca = fma(al, Kh, -d23), al2 = al + al;
    double Auu[6];  // A~^{ab}
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = p; b < 3; ++b) {
        const int q = S(p, b);
        const double v = fma(At[S(p, 2)], Aud[2][b], fma(At[S(p, 1)], Aud[1][b], At[S(p, 0)] * Aud[0][b]));
        Auu[q] = fma(ig[S(p, 2)], Aud[b][2], fma(ig[S(p, 1)], Aud[b][1], ig[S(p, 0)] * Aud[b][0]));
        r0[q] = fma(-al2, v, fma(ca, At[q], fma(cg, gt[q], fma(chi, M[q], sA[q]))));
      }
    AA = fma(2.0, fma(Auu[4], At[4], fma(Auu[2], At[2], Auu[1] * At[1])),
             fma(Auu[5], At[5], fma(Auu[3], At[3], Auu[0] * At[0])));
    double u[3];  // 2 d_b alpha + 3 alpha / chi d_b chi
#pragma unroll
    for (int b = 0; b < 3; ++b) u[b] = fma(3.0 * al2, w[b], dal[b] + dal[b]);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      double r = rGh[p];
#pragma unroll
      for (int b = 0; b < 3; ++b) r = fma(-Auu[S(p, b)], u[b], r);
      const double sd = fma(Gu[p][5], Auu[5], fma(Gu[p][3], Auu[3], Gu[p][0] * Auu[0]));
      const double so = fma(Gu[p][4], Auu[4], fma(Gu[p][2], Auu[2], Gu[p][1] * Auu[1]));
      rGh[p] = fma(al2, fma(2.0, so, sd), r);
    }
  }

  // ---- Khat and Theta
  {
    const double Zdal = 0.5 * chi * fma(y[2], dal[2], fma(y[1], dal[1], y[0] * dal[0]));
    double dK[3], dT[3];
    const double rK = sten.template cross<Z4_DERIV>(7, dK, nullptr);
    const double rT = sten.template cross<Z4_DERIV>(17, dT, nullptr);
    double r = fma(-chi, trD, rK);
    r = fma(al, fma((1.0 / 3.0) * Kt, Kt, fma(kz, Th, AA)), r);
    out(7, fma(2.0, Zdal, r), Kh);
    r = fma(chi, trR, -AA);  // R + 2 nabla_i Z^i = chi gt^{ij} (Rhat + Rchi)_ij
    r = fma((2.0 / 3.0) * Kh, Kh, r);
    r = fma((2.0 / 3.0) * Th, fma(-2.0, Th, Kh), r);
    r = fma(0.5 * al, r, rT - Zdal);
    out(17, fma(-2.0 * al * kz, Th, r), Th);
    // the terms of d/dt Gammahat with gt^{ab}: -2/3 alpha (2 d_b Khat + d_b Theta)
    // - 2 Theta d_b alpha
    const double c1 = (-2.0 / 3.0) * al, c2 = -2.0 * Th;
#pragma unroll
    for (int b = 0; b < 3; ++b) dK[b] = fma(c1, fma(2.0, dK[b], dT[b]), c2 * dal[b]);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int b = 0; b < 3; ++b) rGh[p] = fma(ig[S(p, b)], dK[b], rGh[p]);
  }

  // ---- A~, Gammahat (Eq. syseq2), shift and B (Gamma-driver)
#pragma unroll
  for (int q = 0; q < 6; ++q)
    out(8 + q, sten.template cross<Z4_ADV>(8 + q, nullptr, nullptr) + r0[q], At[q]);
#pragma unroll
  for (int p = 0; p < 3; ++p) out(14 + p, GhAK[p] + rGh[p], Gh[p]);
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const double b = src.centre(22 + p);
    if (zc.shift_frozen) {
      out(19 + p, 0.0, sten.be[p]);
      out(22 + p, 0.0, b);
    } else {
      const double r = sten.template cross<Z4_ADV>(22 + p, nullptr, nullptr);
      out(19 + p, fma(zc.g_shift, b, betaAcc[p]), sten.be[p]);
      out(22 + p, fma(-zc.eta, b, r + rGh[p]), b);
    }
  }
}

}  // namespace sf
