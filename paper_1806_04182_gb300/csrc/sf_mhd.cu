// Ideal Newtonian MHD (Sec. IV.B), 8 conserved fields
//   U = (rho, S_x, S_y, S_z, E, B^x, B^y, B^z),
// in conservative form L(U)_i = -sum_d (F_{i+1/2} - F_{i-1/2}) / dx_d (Eq. 5).
// Interface fluxes: WENO reconstruction of the evolved fields from the left
// and right (WENO5 with JS or Z weights, App. B; WENO3, App. A), physical
// fluxes of both states and the local Lax-Friedrichs formula (Eq. LLF) with
// the largest fast magnetosonic signal speed of the two states; or, with
// flux_split, the same reconstructions applied to the Lax-Friedrichs split
// fluxes.  Fused with the RK stage update.
#include "sf_mhd.cuh"

namespace sf {

// App. B smoothness indicators of the three WENO5 stencils of cell c, from
// w[0..4] = U_{c-2..c+2}: beta_0 of cells c..c+2, beta_1 of c-1..c+1, beta_2
// of c-2..c.  They measure the candidate polynomials on cell c, so the
// reconstructions at both edges of the cell use the same three numbers.
template <typename T>
__device__ __forceinline__ void weno5_beta(const T* w, T& be0, T& be1, T& be2) {
  const T a0 = w[2] - T(2) * w[3] + w[4], b0 = T(3) * w[2] - T(4) * w[3] + w[4];
  const T a1 = w[1] - T(2) * w[2] + w[3], b1 = w[1] - w[3];
  const T a2 = w[0] - T(2) * w[1] + w[2], b2 = w[0] - T(4) * w[1] + T(3) * w[2];
  be0 = T(13.0 / 12.0) * a0 * a0 + T(0.25) * b0 * b0;
  be1 = T(13.0 / 12.0) * a1 * a1 + T(0.25) * b1 * b1;
  be2 = T(13.0 / 12.0) * a2 * a2 + T(0.25) * b2 * b2;
}

// App. B nonlinear combination of the candidates c_k of stencils k = 0, 1, 2
// with linear weights g_k and smoothness indicators be_k: JS weights
// g_k / (eps + be_k)^2, or with Z the WENO-Z weights g_k (1 + (tau / (eps +
// be_k))^q), tau = |be_0 - be_2|, normalised by their sum.  In double the
// weights are formed over the common denominator (eps + be_0)^2 (eps + be_1)^2
// (eps + be_2)^2 (WENO-Z for q = 2), which cancels in the normalisation: one
// division instead of four (the products of squares would underflow float on
// fine grids, so float keeps the per-weight divisions).
template <typename T, bool Z>
__device__ __forceinline__ T weno5_combine(T c0, T c1, T c2, T g0, T g1, T g2, T be0, T be1, T be2,
                                           T eps, const MhdCoef<T>& mc) {
  T al0, al1, al2;
  if constexpr (Z) {
    const T tau = fabs(be0 - be2);
    if (sizeof(T) == 8 && mc.q == T(2)) {
      const T e0 = eps + be0, e1 = eps + be1, e2 = eps + be2, t2 = tau * tau;
      const T q0 = e0 * e0, q1 = e1 * e1, q2 = e2 * e2;
      al0 = g0 * (q0 + t2) * (q1 * q2);
      al1 = g1 * (q1 + t2) * (q0 * q2);
      al2 = g2 * (q2 + t2) * (q0 * q1);
    } else {
      al0 = g0 * (T(1) + wz_pow(tau / (eps + be0), mc.q));
      al1 = g1 * (T(1) + wz_pow(tau / (eps + be1), mc.q));
      al2 = g2 * (T(1) + wz_pow(tau / (eps + be2), mc.q));
    }
  } else if constexpr (sizeof(T) == 8) {
    const T e0 = eps + be0, e1 = eps + be1, e2 = eps + be2;
    const T q0 = e0 * e0, q1 = e1 * e1, q2 = e2 * e2;
    al0 = g0 * (q1 * q2);
    al1 = g1 * (q0 * q2);
    al2 = g2 * (q0 * q1);
  } else {
    const T e0 = eps + be0, e1 = eps + be1, e2 = eps + be2;
    al0 = g0 / (e0 * e0);
    al1 = g1 / (e1 * e1);
    al2 = g2 / (e2 * e2);
  }
  return (al0 * c0 + al1 * c1 + al2 * c2) / (al0 + al1 + al2);
}

// App. B: left state at i+1/2 (the right edge of cell i) from w[0..4] =
// U_{i-2..i+2}; Z: WENO-Z weights
template <typename T, bool Z>
__device__ __forceinline__ T weno_left(const T* w, T eps, const MhdCoef<T>& mc) {
  const T c0 = (T(2) * w[2] + T(5) * w[3] - w[4]) * T(1.0 / 6.0);
  const T c1 = (-w[1] + T(5) * w[2] + T(2) * w[3]) * T(1.0 / 6.0);
  const T c2 = (T(2) * w[0] - T(7) * w[1] + T(11) * w[2]) * T(1.0 / 6.0);
  T be0, be1, be2;
  weno5_beta(w, be0, be1, be2);
  return weno5_combine<T, Z>(c0, c1, c2, T(0.3), T(0.6), T(0.1), be0, be1, be2, eps, mc);
}

// App. B: right state at i-1/2 (the left edge of cell i) from w[0..4] =
// U_{i-2..i+2}; Z: WENO-Z weights
template <typename T, bool Z>
__device__ __forceinline__ T weno_right(const T* w, T eps, const MhdCoef<T>& mc) {
  const T c0 = (T(2) * w[4] - T(7) * w[3] + T(11) * w[2]) * T(1.0 / 6.0);
  const T c1 = (-w[3] + T(5) * w[2] + T(2) * w[1]) * T(1.0 / 6.0);
  const T c2 = (T(2) * w[2] + T(5) * w[1] - w[0]) * T(1.0 / 6.0);
  T be0, be1, be2;
  weno5_beta(w, be0, be1, be2);
  return weno5_combine<T, Z>(c0, c1, c2, T(0.1), T(0.6), T(0.3), be0, be1, be2, eps, mc);
}

// App. A: WENO3 left state at i+1/2 from w[1..3] = U_{i-1..i+1}
template <typename T>
__device__ __forceinline__ T weno3_left(const T* w, T eps) {
  const T c0 = T(0.5) * w[2] + T(0.5) * w[3];
  const T c1 = T(-0.5) * w[1] + T(1.5) * w[2];
  const T b0 = (w[3] - w[2]) * (w[3] - w[2]);
  const T b1 = (w[2] - w[1]) * (w[2] - w[1]);
  const T e0 = eps + b0, e1 = eps + b1;
  if constexpr (sizeof(T) == 8) {  // common denominator e0^2 e1^2 (see weno5_combine)
    const T a0 = T(2.0 / 3.0) * (e1 * e1), a1 = T(1.0 / 3.0) * (e0 * e0);
    return (a0 * c0 + a1 * c1) / (a0 + a1);
  }
  const T a0 = T(2.0 / 3.0) / (e0 * e0), a1 = T(1.0 / 3.0) / (e1 * e1);
  return (a0 * c0 + a1 * c1) / (a0 + a1);
}

// App. A: WENO3 right state at i-1/2 from w[1..3] = U_{i-1..i+1}
template <typename T>
__device__ __forceinline__ T weno3_right(const T* w, T eps) {
  const T c0 = T(-0.5) * w[3] + T(1.5) * w[2];
  const T c1 = T(0.5) * w[2] + T(0.5) * w[1];
  const T b0 = (w[2] - w[3]) * (w[2] - w[3]);
  const T b1 = (w[1] - w[2]) * (w[1] - w[2]);
  const T e0 = eps + b0, e1 = eps + b1;
  if constexpr (sizeof(T) == 8) {  // common denominator e0^2 e1^2 (see weno5_combine)
    const T a0 = T(1.0 / 3.0) * (e1 * e1), a1 = T(2.0 / 3.0) * (e0 * e0);
    return (a0 * c0 + a1 * c1) / (a0 + a1);
  }
  const T a0 = T(1.0 / 3.0) / (e0 * e0), a1 = T(2.0 / 3.0) / (e1 * e1);
  return (a0 * c0 + a1 * c1) / (a0 + a1);
}

// one of three values by a direction d that may be known only at run time
// (selects, not an indexed array, so that nothing goes to local memory)
template <typename T>
__device__ __forceinline__ T by_dir(int d, T x, T y, T z) {
  return d == 0 ? x : (d == 1 ? y : z);
}

// physical flux along d and the largest signal speed |v_d| + c_fast,d
template <typename T>
__device__ __forceinline__ T flux_speed(const T* q, int d, const MhdCoef<T>& mc, T* F) {
  const T rho = q[0], irho = T(1) / rho;
  const T v[3] = {q[1] * irho, q[2] * irho, q[3] * irho};
  const T B[3] = {q[5], q[6], q[7]};
  const T B2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
  const T S2v = q[1] * v[0] + q[2] * v[1] + q[3] * v[2];
  const T pr = (mc.gamma - T(1)) * (q[4] - T(0.5) * S2v - T(0.5) * B2);
  const T ptot = pr + T(0.5) * B2;
  const T vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2];
  const T vd = by_dir(d, v[0], v[1], v[2]), Bd = by_dir(d, B[0], B[1], B[2]);
  const T Sd = by_dir(d, q[1], q[2], q[3]);
  F[0] = Sd;
#pragma unroll
  for (int a = 0; a < 3; ++a) F[1 + a] = Sd * v[a] - Bd * B[a] + (a == d ? ptot : T(0));
  F[4] = (q[4] + ptot) * vd - vB * Bd;
#pragma unroll
  for (int a = 0; a < 3; ++a) F[5 + a] = vd * B[a] - v[a] * Bd;
  const T a2 = mc.gamma * pr * irho, b2 = B2 * irho, bd2 = Bd * Bd * irho;
  const T s = a2 + b2;
  const T cf2 = T(0.5) * (s + sqrt(s * s - T(4) * a2 * bd2));
  return fabs(vd) + sqrt(cf2);
}

// Flux through the same face from the reconstruction of the split fluxes
// (Sec. II.B.2, Lax-Friedrichs splitting): S = the largest signal speed over
// the six cells p-2..p+3, F+- = (F(U) +- S U)/2 at each cell, F+ reconstructed
// from the left (cells p-2..p+2) plus F- from the right (cells p-1..p+3).
template <typename T, int VAR>
__device__ __forceinline__ void face_flux_split(const T* p, long long F, long long s,
                                                int d, const MhdCoef<T>& mc, T* Fout) {
  const T eps = by_dir(d, mc.eps[0], mc.eps[1], mc.eps[2]);
  T Uc[6][8], Fc[6][8];
  T S = T(0);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
#pragma unroll
    for (int f = 0; f < 8; ++f) Uc[c][f] = p[f * F + (c - 2) * s];
    const T sp = flux_speed(Uc[c], d, mc, Fc[c]);
    S = sp > S ? sp : S;
  }
#pragma unroll
  for (int f = 0; f < 8; ++f) {
    T wp[6], wm[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      wp[c] = T(0.5) * (Fc[c][f] + S * Uc[c][f]);
      wm[c] = T(0.5) * (Fc[c][f] - S * Uc[c][f]);
    }
    if constexpr (VAR == 2)
      Fout[f] = weno3_left(wp, eps) + weno3_right(wm + 1, eps);
    else
      Fout[f] = weno_left<T, VAR == 1>(wp, eps, mc) + weno_right<T, VAR == 1>(wm + 1, eps, mc);
  }
}

// ------------------------------------------------------------ stage kernels
// The largest signal rate of a block's outputs into *rate: block max, then
// one atomic per block (non-negative doubles order as their bits).
template <int NW>
__device__ __forceinline__ void block_rate(double rate, double* s_rate, double* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rate = fmax(rate, __shfl_down_sync(0xffffffffu, rate, o));
  if (threadIdx.x == 0) s_rate[threadIdx.y] = rate;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    double m = 0.0;
    for (int w = 0; w < NW; ++w) m = fmax(m, s_rate[w]);
    atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(m));
  }
}

// max over d of (|v_d| + c_fast,d) / dx_d of a cell, 0 if that is no number.
// float: kept in float, whose maximum is the same number without conversions
// and comparisons on the FP64 pipe.  double: the operations of llf_flux2, 73 on
// that pipe where the IEEE quotients and six IEEE roots make it about 160, and
// rounded explicitly, so that both of its callers get the same bits.
__device__ __forceinline__ float cell_rate(const float* q, const MhdCoef<float>& mc) {
  float rate = 0.0f, Fd[8];
#pragma unroll
  for (int d = 0; d < 3; ++d) rate = fmaxf(rate, flux_speed(q, d, mc, Fd) * mc.idx[d]);
  return rate;
}
__device__ __forceinline__ double cell_rate(const double* q, const MhdCoef<double>& mc) {
  const double nir = nrecip1<false>(q[0]);
  const double* b = q + 5;
  double nv[3], bb[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    nv[d] = __dmul_rn(q[1 + d], nir);
    bb[d] = __dmul_rn(b[d], b[d]);
  }
  const double B2 = __dadd_rn(__dadd_rn(bb[0], bb[1]), bb[2]);
  const double nSvB = __fma_rn(q[3], nv[2], __fma_rn(q[2], nv[1], __fma_rn(q[1], nv[0], -B2)));
  const double pr = __dmul_rn(__dsub_rn(mc.gamma, 1.0), __fma_rn(0.5, nSvB, q[4]));
  const double na2 = __dmul_rn(__dmul_rn(mc.gamma, pr), nir);
  const double h = __dmul_rn(-0.5, __fma_rn(B2, nir, na2)), hh = __dmul_rn(h, h);
  const double n2 = -__dmul_rn(na2, nir);
  double rate = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double disc = __fma_rn(n2, bb[d], hh);
    const double cf = sqrt1(nonneg(__dadd_rn(sqrt1(nonneg(disc)), h)));
    rate = fmax(rate, __dmul_rn(__dadd_rn(fabs(nv[d]), cf), mc.idx[d]));  // NaN kept out
  }
  return rate;
}

// The SSP-RK3 stage write of a cell's 8 fields (stage_combine, with the stage
// chosen once for all of them); q receives the new values.
template <typename T>
__device__ __forceinline__ void ssp_write(const PatchArgs<T>& a, const StageArgs& s, const Images& im,
                                          long long c, const T* cen, const T* un_m, const T* r, T* q) {
  T un[8];
#pragma unroll
  for (int f = 0; f < 8; ++f) un[f] = s.un_alias ? cen[f] : un_m[f];
  if (s.stage == 0) {
#pragma unroll
    for (int f = 0; f < 8; ++f) q[f] = un[f] + a.dt * r[f];
  } else if (s.stage == 1) {
#pragma unroll
    for (int f = 0; f < 8; ++f) q[f] = T(0.75) * un[f] + T(0.25) * (cen[f] + a.dt * r[f]);
  } else {
#pragma unroll
    for (int f = 0; f < 8; ++f) q[f] = un[f] * T(1.0 / 3.0) + T(2.0 / 3.0) * (cen[f] + a.dt * r[f]);
  }
  bool bad = false;
#pragma unroll
  for (int f = 0; f < 8; ++f) {
    a.nx[f * a.sf + c] = q[f];
    bad = bad || !finite_(q[f]);
  }
  if (s.check_finite && bad) atomicOr(s.status, ST_NONFINITE);
  if (im.mask) {
#pragma unroll 1
    for (int f = 0; f < 8; ++f) store_images(a, im, f * a.sf + c, a.nx[f * a.sf + c]);
  }
}

// Reconstruction of the evolved fields.  A block of MR + 1 warps owns a column
// of 32 x MR cells per plane and marches in z.  In each of its three
// directions a cell is reconstructed once, both edges together (weno_edges),
// and each face flux is evaluated once: warp w < MR takes row w, the last warp
// the cells and faces that the block's rows need from outside,
//   x: right-edge values of the cells left of the tile (lanes 0 .. MR - 1),
//      left-edge values of the cells right of it (lanes MR .. 2 MR - 1), whose
//      faces it evaluates;
//   y: the row below the tile, the row above it and the face row between;
// so that all 32 x MR cells produce output.  Edge values cross to the next
// cell by shuffle (x), shared memory (y) and in registers along the march
// (z); fluxes likewise.  The last warp's work is a row's (3 reconstructions,
// 2 fluxes), and every warp runs the same instructions with its own pointers,
// so a cell's result does not depend on where in a block it lies.  Before
// the first plane two passes evaluate only z (the right edge of the cell
// below, then the face below the first plane).
//
// double is bound by the FP64 pipe (one warp instruction per 16 cycles and
// SM; 86% busy) and reads its stencils from global memory.  float is bound by
// issue and latency (issue 48%, then fixed-latency waits): its planes are
// staged in shared memory as field pairs by cp.async, five in a ring, so that
// a stencil value pair is one 64-bit load with a constant offset.  MR + 1 is
// 16 or 8: registers are split over the four schedulers, so 9 warps get 168
// each where 8 get 255 (float, 9 warps: 1410 us per 128^3 step, 8: 1155).
// 128^3 SSP-RK3 step with CFL rate, against a kernel that reconstructed each
// cell once per face and side in tiles of 31 x 11 (float) and 31 x 7 outputs:
// double 54.4 -> 20.8 ms, float 2.23 -> 0.92 ms.
//
// A block's work is one chunk of mz planes of one column of tiles or, in
// double where that is less, an even share of all columns laid end to end,
// whose boundaries fall between planes: a launch of as many blocks as the GPU
// holds, all ending together (128^3: 36 columns of 128 planes over 152 SMs,
// 20.9 -> 20.3 ms when a field took 41 operations).  float keeps to chunks:
// the loop over the columns of a share costs registers that its planes need
// (915 -> 965 us).
constexpr int MX = 32;
struct MhdWork {
  int mz;      // planes of a chunk; 0: even shares
  int nx, ny;  // tiles along x and y
};
template <typename T, int MR>
struct MhdSmem {
  static constexpr bool kStaged = sizeof(T) == 4;
  static constexpr int kCols = MX + 6, kCells = kCols * (MR + 6);  // a plane with its halo
  static constexpr int kSlots = 5;
  using P = typename PairOf<T>::type;
  T ey[MR + 1][8][MX];  // right-edge values along y of rows -1 .. MR - 1
  T fy[MR + 1][8][MX];  // y fluxes below rows 0 .. MR
  T exl[8][MR], exr[8][MR], fxr[8][MR];  // x: right edges of cells -1 and 31, flux at 32
  double rate[MR + 1];
  int work[2], end[2];
  P ring[kStaged ? kSlots : 1][kStaged ? 4 * kCells : 1];  // planes as field pairs
};

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One tile's planes k0 .. k1 - 1; the signal rate of the outputs into rate.
template <typename T, int VAR, int MR>
__device__ __forceinline__ void mhd_march(const PatchArgs<T>& a, const StageArgs& s,
                                          const MhdCoef<T>& mc, MhdSmem<T, MR>& sm, int x0, int y0,
                                          int k0, int k1, T& rate) {
  using S = MhdSmem<T, MR>;
  using P = typename S::P;
  constexpr int NC = S::kCells, CW = S::kCols;
  constexpr bool ST = S::kStaged;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const bool row = ty < MR;
  const int g = a.g;
  const int i = x0 + tx, j = y0 + ty;
  const bool out = row && i < a.n[0] && j < a.n[1];
  const int xr = tx % MR;                  // the last warp's x lanes: their row,
  const bool xright = (tx / MR) % 2 == 1;  // and which side of the tile
  const bool do_xz = !row || j < a.n[1], do_y = !row || j <= a.n[1];
  const int ys = row ? ty + 1 : 0, yl = row ? ty : MR;  // ey rows written / read, fy row written
  // cell offsets in a plane (x, y and third reconstruction), in the staged
  // plane or in the global one.  Cells outside the patch that a face needs lie
  // in its ghost zone; lanes and rows beyond those repeat others (their
  // results go nowhere).
  long long gx = 0, gy = 0, gz = 0;
  int lx_ = 0, ly_ = 0, lz_ = 0;
  const long long c0 = (long long)(min(j, a.n[1]) + g) * a.sy + (min(i, a.n[0]) + g);
  if constexpr (ST) {
    ly_ = ((row ? ty : -1) + 3) * CW + tx + 3;
    lx_ = row ? ly_ : (xr + 3) * CW + (xright ? MX : -1) + 3;
    lz_ = row ? ly_ : (MR + 3) * CW + tx + 3;
  } else {
    auto cell = [&](int ci, int cj) {
      return (long long)(min(cj, a.n[1]) + g) * a.sy + (min(ci, a.n[0]) + g);
    };
    gy = row ? c0 : cell(i, y0 - 1);
    gx = row ? c0 : cell(xright ? x0 + MX : x0 - 1, y0 + xr);
    gz = row ? c0 : cell(i, y0 + MR);
  }
  // staging: plane p (interior index) into ring slot q, each thread its cells
  constexpr int NT = MX * (MR + 1), NS = (NC + NT - 1) / NT;
  long long so[NS];
  if constexpr (ST) {
#pragma unroll
    for (int e = 0; e < NS; ++e) {
      const int t = ty * MX + tx + e * NT;
      const int cx = min(x0 - 3 + t % CW, a.n[0] + 2), cy = min(y0 - 3 + t / CW, a.n[1] + 2);
      so[e] = (long long)(cy + g) * a.sy + (cx + g);
    }
  }
  auto stage = [&](int p, int q) {
    if constexpr (ST) {
      const T* pl = a.us + (long long)(p + g) * a.sz;
#pragma unroll
      for (int e = 0; e < NS; ++e) {
        const int t = ty * MX + tx + e * NT;
        if (t < NC) {
          const T* src = pl + so[e];
          float* dst = reinterpret_cast<float*>(&sm.ring[q][t]);
#pragma unroll
          for (int f = 0; f < 8; ++f, src += a.sf) cp_async4(dst + (f / 2) * (2 * NC) + f % 2, src);
        }
      }
    }
  };
  // (left, right) states of a face
  auto states = [](const P* l, const P* r, P* q) {
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      q[2 * f] = P(l[f].x, r[f].x);
      q[2 * f + 1] = P(l[f].y, r[f].y);
    }
  };
  P erz[4];           // right-edge values along z of the cell below
  T Fzm[8];           // z flux below the current plane
#pragma unroll
  for (int f = 0; f < 4; ++f) erz[f] = P(T(1));
  int sl[5] = {0, 1, 2, 3, 4};  // ring slots of planes k - 1 .. k + 3
  if constexpr (ST) {
    for (int q = 0; q < 5; ++q) stage(k0 - 3 + q, q);
    cp_async_wait();
    __syncthreads();
  }
  for (int k = k0 - 2; k < k1; ++k) {
    const T* plane = a.us + (long long)(k + g) * a.sz;
    const bool body = k >= k0;
    // both edges of a cell from the plane's values at stride st (staged: cells
    // of the ring slot of plane k; global: elements)
    auto recon = [&](int lc, long long gc, int lst, long long gst, T eps, P* er, P* el) {
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        P w[5];
#pragma unroll
        for (int o = 0; o < 5; ++o) {
          if constexpr (ST) {
            w[o] = sm.ring[sl[1]][f * NC + lc + (o - 2) * lst];
          } else {
            const T* q = plane + gc + (o - 2) * gst + 2 * f * a.sf;
            w[o] = P(*q, q[a.sf]);
          }
        }
        weno_edges<VAR, T, P>(w, eps, mc, er[f], el[f]);
      }
    };
    P rx[4], lx[4], ly[4];
    T dz[8];
    if (body && do_y) {
      P ry[4];
      recon(ly_, gy, CW, a.sy, mc.eps[1], ry, ly);
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        sm.ey[ys][2 * f][tx] = ry[f].x;
        sm.ey[ys][2 * f + 1][tx] = ry[f].y;
      }
    }
    if (body && do_xz) {
      recon(lx_, gx, 1, 1, mc.eps[0], rx, lx);
      if (row && tx == MX - 1) {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          sm.exr[2 * f][ty] = rx[f].x;
          sm.exr[2 * f + 1][ty] = rx[f].y;
        }
      }
      if (!row && tx < MR) {
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          sm.exl[2 * f][tx] = rx[f].x;
          sm.exl[2 * f + 1][tx] = rx[f].y;
        }
      }
    }
    if (do_xz && (row || body)) {
      // rows: cell k + 1 along z; the last warp: the row above the tile along y
      P r[4], l[4];
      const T eps = row ? mc.eps[2] : mc.eps[1];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        P w[5];
#pragma unroll
        for (int o = 0; o < 5; ++o) {
          if constexpr (ST) {
            w[o] = sm.ring[row ? sl[o] : sl[1]][f * NC + lz_ + (row ? 0 : (o - 2) * CW)];
          } else {
            const T* q = plane + (row ? a.sz : 0) + gz + (o - 2) * (row ? a.sz : a.sy) + 2 * f * a.sf;
            w[o] = P(*q, q[a.sf]);
          }
        }
        weno_edges<VAR, T, P>(w, eps, mc, r[f], l[f]);
      }
      if (row) {
        P q[8];
        T F[8];
        states(erz, l, q);
        llf_flux2<2, T, P>(q, mc.gamma, F);
#pragma unroll
        for (int f = 0; f < 8; ++f) {
          dz[f] = F[f] - Fzm[f];
          Fzm[f] = F[f];
        }
#pragma unroll
        for (int f = 0; f < 4; ++f) erz[f] = r[f];
      } else {
#pragma unroll
        for (int f = 0; f < 4; ++f) ly[f] = l[f];
      }
    }
    if (body || ST) __syncthreads();  // ey, exl, exr; plane k - 1 is read
    if constexpr (ST) {
      if (k + 1 < k1) stage(k + 4, sl[0]);
    }
    if (body) {
      T Fx[8], Fy[8];
      if (do_xz) {
        P lt[4], q[8];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          lt[f].x = __shfl_up_sync(0xffffffffu, rx[f].x, 1);
          lt[f].y = __shfl_up_sync(0xffffffffu, rx[f].y, 1);
        }
        if (row ? tx == 0 : xright) {
#pragma unroll
          for (int f = 0; f < 4; ++f)
            lt[f] = row ? P(sm.exl[2 * f][ty], sm.exl[2 * f + 1][ty])
                        : P(sm.exr[2 * f][xr], sm.exr[2 * f + 1][xr]);
        }
        states(lt, lx, q);
        llf_flux2<0, T, P>(q, mc.gamma, Fx);
        if (!row && xright) {
#pragma unroll
          for (int f = 0; f < 8; ++f) sm.fxr[f][xr] = Fx[f];
        }
      }
      if (do_y) {
        P lt[4], q[8];
#pragma unroll
        for (int f = 0; f < 4; ++f) lt[f] = P(sm.ey[yl][2 * f][tx], sm.ey[yl][2 * f + 1][tx]);
        states(lt, ly, q);
        llf_flux2<1, T, P>(q, mc.gamma, Fy);
#pragma unroll
        for (int f = 0; f < 8; ++f) sm.fy[yl][f][tx] = Fy[f];
      }
      // U^n, if a stage reads it from memory, on its way across the barrier
      const long long c = (long long)(k + g) * a.sz + c0;
      T un[8];
      if (!s.un_alias && s.mode == 0 && out) {
#pragma unroll
        for (int f = 0; f < 8; ++f) un[f] = a.un[f * a.sf + c];
      }
      if constexpr (ST) cp_async_wait();
      __syncthreads();  // fy, fxr; plane k + 4
      if (row && do_xz) {
        T q[8], rhs[8];
#pragma unroll
        for (int f = 0; f < 8; ++f) {
          T fxp = __shfl_down_sync(0xffffffffu, Fx[f], 1);
          if (tx == MX - 1) fxp = sm.fxr[f][ty];
          // the fluxes are twice the fluxes
          T r = (fxp - Fx[f]) * (T(-0.5) * mc.idx[0]);
          r = fma(sm.fy[ty + 1][f][tx] - Fy[f], T(-0.5) * mc.idx[1], r);
          r = fma(dz[f], T(-0.5) * mc.idx[2], r);
          rhs[f] = r;
        }
        if (out) {
          T cen[8];
#pragma unroll
          for (int f = 0; f < 8; ++f) {
            if constexpr (ST) {
              const P v = sm.ring[sl[1]][(f / 2) * NC + lz_];
              cen[f] = f % 2 ? v.y : v.x;
            } else {
              cen[f] = a.us[f * a.sf + c];
            }
          }
          const Images im = ghost_images(a, s, i, j, k);
          if (s.mode == 0 && s.rk == SF_SSPRK3)
            ssp_write(a, s, im, c, cen, un, rhs, q);
          else
#pragma unroll
            for (int f = 0; f < 8; ++f) q[f] = write_field(a, s, im, f, c, i, j, k, cen[f], rhs[f]);
        }
        if (out && a.rate) rate = fmax(rate, cell_rate(q, mc));
      }
    } else if constexpr (ST) {
      cp_async_wait();
      __syncthreads();
    }
    const int t = sl[0];
#pragma unroll
    for (int q = 0; q < 4; ++q) sl[q] = sl[q + 1];
    sl[4] = t;
  }
}

template <typename T, int VAR, int MR>
__global__ void __launch_bounds__(MX * (MR + 1), 16 / (MR + 1))
    mhd_stage_kernel(PatchArgs<T> a, StageArgs s, MhdCoef<T> mc, MhdWork wk) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MhdSmem<T, MR>& sm = *reinterpret_cast<MhdSmem<T, MR>*>(smem_raw);
  wait_predecessor();
  const bool even = sizeof(T) == 8 && wk.mz == 0, first = threadIdx.x == 0 && threadIdx.y == 0;
  T rate = 0;  // max signal rate of this thread's outputs (fused CFL reduction)
  // an even share goes from plane work[1] of column work[0] to before plane
  // end[1] of column end[0] (in shared memory: the march has no registers to spare)
  if (even) {
    if (first) {
      const int len = 3 * a.n[2] + 2;  // a column in thirds of a plane
      const long long total = (long long)wk.nx * wk.ny * len;
      // the first plane that starts at or after boundary b
      auto cut = [&](unsigned b, int& c, int& k) {
        const long long at = total * b / gridDim.x;
        c = (int)(at / len);
        k = ((int)(at - (long long)c * len) + 2) / 3;
        if (k >= a.n[2]) {
          k = 0;
          ++c;
        }
      };
      cut(blockIdx.x, sm.work[0], sm.work[1]);
      cut(blockIdx.x + 1, sm.end[0], sm.end[1]);
    }
    __syncthreads();
  }
#pragma unroll 1
  while (true) {
    int bx = blockIdx.x, by = blockIdx.y, k0 = blockIdx.z * wk.mz, k1 = min(k0 + wk.mz, a.n[2]);
    if (even) {
      const int col = sm.work[0], last = sm.end[0];
      k0 = sm.work[1];
      k1 = col == last ? sm.end[1] : a.n[2];
      if (col > last || k0 >= k1) break;
      bx = col % wk.nx;
      by = col / wk.nx;
    }
    mhd_march<T, VAR, MR>(a, s, mc, sm, bx * MX, by * MR, k0, k1, rate);
    if (!even) break;
    __syncthreads();  // the next column reuses the shared arrays
    if (first) {
      ++sm.work[0];
      sm.work[1] = 0;
    }
    __syncthreads();
  }
  if (a.rate) block_rate<MR + 1>(rate, sm.rate, a.rate);
}

// Lax-Friedrichs flux splitting.  The split fluxes of a cell depend on the
// face (S is the face's), so both sides are reconstructed per face: a block of
// 32 x 8 threads owns 31 x 7 output cells of a plane; thread (tx, ty)
// evaluates the x-face at i - 1/2 and the y-face at j - 1/2 of its column, so
// the +1/2 faces of the output cells come from lane tx + 1 (warp shuffle) and
// row ty + 1 (shared memory), and carries the z-face below the current plane
// in registers while it marches mz planes (a first pass evaluates only the
// z-face below the first plane).  The three directions run in one rolled
// loop, so the kernel holds one copy of the face code.  One block per SM is
// asked for (without that the compiler halves the reads in flight of float
// WENO5: 20^3 WENO-Z step 413 against 430 us), two for float WENO3, which fits
// in 128 registers (110 x 30 x 70 step 467 -> 319 us).
constexpr int SY = 8;
template <typename T, int VAR>
__global__ void __launch_bounds__(MX * SY, sizeof(T) == 4 && VAR == 2 ? 2 : 1)
    mhd_split_kernel(PatchArgs<T> a, StageArgs s, MhdCoef<T> mc, int mz) {
  __shared__ T fy[SY][MX][8];
  wait_predecessor();
  __shared__ double s_rate[SY];
  const int tx = threadIdx.x, ty = threadIdx.y;
  double rate = 0.0;  // max signal rate of this thread's outputs (fused CFL reduction)
  const int i = blockIdx.x * (MX - 1) + tx;
  const int j = blockIdx.y * (SY - 1) + ty;
  const int k0 = blockIdx.z * mz;
  const int k1 = min(k0 + mz, a.n[2]);
  const int g = a.g;
  const bool out = tx < MX - 1 && ty < SY - 1 && i < a.n[0] && j < a.n[1];
  const bool xface = i <= a.n[0] && j < a.n[1];
  const bool yface = j <= a.n[1] && i < a.n[0];
  auto at = [&](int ii, int jj, int kk) {
    return a.us + (long long)(kk + g) * a.sz + (long long)(jj + g) * a.sy + (ii + g);
  };
  T Fzm[8];
  // pass k = k0 - 1 evaluates only the z-face below the first plane (Fzm);
  // `body` is the same for the whole block, so the barriers below are taken
  // by every thread or by none
  for (int k = k0 - 1; k < k1; ++k) {
    const bool body = k >= k0;
    T Fx[8], Fy[8], Fz[8];
#pragma unroll 1
    for (int d = body ? 0 : 2; d < 3; ++d) {
      T Fd[8];
      if (d == 0 ? xface : (d == 1 ? yface : out)) {
        const T* base = d == 0 ? at(i - 1, j, k) : (d == 1 ? at(i, j - 1, k) : at(i, j, k));
        face_flux_split<T, VAR>(base, a.sf, d == 0 ? 1LL : (d == 1 ? a.sy : a.sz), d, mc, Fd);
      } else {
#pragma unroll
        for (int f = 0; f < 8; ++f) Fd[f] = T(0);
      }
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        Fx[f] = d == 0 ? Fd[f] : Fx[f];
        Fy[f] = d == 1 ? Fd[f] : Fy[f];
        Fz[f] = d == 2 ? Fd[f] : Fz[f];
      }
    }
    if (!body) {
#pragma unroll
      for (int f = 0; f < 8; ++f) Fzm[f] = Fz[f];
      continue;
    }
#pragma unroll
    for (int f = 0; f < 8; ++f) fy[ty][tx][f] = Fy[f];
    T Fxp[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) Fxp[f] = __shfl_down_sync(0xffffffffu, Fx[f], 1);
    __syncthreads();
    if (out) {
      const long long c = (long long)(k + g) * a.sz + (long long)(j + g) * a.sy + (i + g);
      const Images im = ghost_images(a, s, i, j, k);
      T q[8];
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        T r = T(0);
        r -= (Fxp[f] - Fx[f]) * mc.idx[0];
        r -= (fy[ty + 1][tx][f] - Fy[f]) * mc.idx[1];
        r -= (Fz[f] - Fzm[f]) * mc.idx[2];
        q[f] = write_field(a, s, im, f, c, i, j, k, a.us[f * a.sf + c], r);
        Fzm[f] = Fz[f];
      }
      if (a.rate) rate = fmax(rate, cell_rate(q, mc));
    }
    __syncthreads();
  }
  if (a.rate) block_rate<SY>(rate, s_rate, a.rate);
}

// CFL rate: max over cells and d of (|v_d| + c_fast,d) / dx_d
template <typename T>
__global__ void __launch_bounds__(256) mhd_rate_kernel(const T* __restrict__ u0, int nx, int ny,
                                                       int nz, int g, long long sy, long long sz,
                                                       long long F, MhdCoef<T> mc,
                                                       unsigned long long* out) {
  const long long total = (long long)nx * ny * nz;
  double best = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % nx);
    const int j = (int)((t / nx) % ny);
    const int k = (int)(t / ((long long)nx * ny));
    const T* p = u0 + (long long)(k + g) * sz + (long long)(j + g) * sy + (i + g);
    T q[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) q[f] = __ldg(p + f * F);
    if constexpr (sizeof(T) == 8) {
      best = fmax(best, cell_rate(q, mc));
    } else {
      T Fd[8];
#pragma unroll
      for (int d = 0; d < 3; ++d) best = fmax(best, double(flux_speed(q, d, mc, Fd)) * double(mc.idx[d]));
    }
  }
  // block max, then one atomic per block (non-negative doubles order like their bits)
  __shared__ double sm[256];
  sm[threadIdx.x] = best;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicMax(out, (unsigned long long)__double_as_longlong(sm[0]));
}

template <typename T>
static MhdCoef<T> coef(const sf_params& prm, const sf_patch& p) {
  MhdCoef<T> mc;
  mc.gamma = T(prm.gamma_eos);
  for (int d = 0; d < 3; ++d) {
    const double h = p.dx[d];
    mc.eps[d] = T(prm.weno_eps > 0 ? prm.weno_eps
                                   : (prm.weno_variant == 2 ? h * h : h * h * h * h));
    mc.idx[d] = T(1.0 / h);
  }
  mc.q = T(prm.weno_q);
  mc.variant = prm.weno_variant;
  mc.split = prm.flux_split;
  return mc;
}

// Planes per block along z: a block evaluates mz planes and the passes before
// its first one, about (3 mz + extra) / 3 planes' work, and a launch of B
// blocks takes ceil(B / resident) rounds of the resident blocks (blocks per
// SM x SMs), so mz in [lo, hi] minimises the cost ceil(B(mz) / resident)
// (3 mz + extra); ties go to the larger mz.  The split kernel, which reads its
// stencils from global memory, keeps to 4 .. 16 planes (99 x 48 x 88 float in 1
// .. 32: 1036 instead of 1021 us).  Only chunk lengths whose grid fits gridDim.z
// (65535) are considered.
struct MhdPlan {
  int mz;  // 0: even shares over `resident` blocks
  long long cost;
};
static MhdPlan mhd_planes_per_block(int gx, int gy, int nz, int resident, int extra, int lo, int hi) {
  MhdPlan best = {hi, -1};
  for (int mz = hi; mz >= lo; --mz) {
    if ((nz + mz - 1) / mz > 65535) break;
    const long long blocks = (long long)gx * gy * ((nz + mz - 1) / mz);
    const long long rounds = resident > 0 ? (blocks + resident - 1) / resident : blocks;
    const long long cost = rounds * (3 * mz + extra);
    if (best.cost < 0 || cost < best.cost) best = {mz, cost};
  }
  return best;
}

// A stage kernel instance: block, tile of output cells and dynamic shared
// memory.  ROWS: the output rows of mhd_stage_kernel, 0 for mhd_split_kernel.
template <typename T, int VAR, int ROWS>
struct MhdInstance {
  static constexpr int threads_y = ROWS ? ROWS + 1 : SY;
  static constexpr int out_x = ROWS ? MX : MX - 1, out_y = ROWS ? ROWS : SY - 1;
  static constexpr int smem = ROWS ? (int)sizeof(MhdSmem<T, ROWS ? ROWS : 1>) : 0;
  static constexpr auto kernel() {
    if constexpr (ROWS == 0)
      return mhd_split_kernel<T, VAR>;
    else
      return mhd_stage_kernel<T, VAR, ROWS>;
  }
  // Resident blocks on the current device (blocks per SM x SMs), cached per
  // device; 0 if unknown.  The first call on a device opts the kernel into
  // its shared memory.
  static int resident() {
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (!cache[dev]) {
      int per_sm = 0, sms = 0;
      if (cudaFuncSetAttribute(kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel(), MX * threads_y, smem) !=
              cudaSuccess ||
          cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
      cache[dev] = per_sm * sms;
    }
    return cache[dev];
  }
  static MhdPlan plan(const sf_patch& p) {
    const MhdPlan chunks = mhd_planes_per_block((p.n[0] + out_x - 1) / out_x,
                                                (p.n[1] + out_y - 1) / out_y, p.n[2], resident(),
                                                ROWS ? 2 : 1, ROWS ? 1 : 4, ROWS ? 32 : 16);
    if (!ROWS || sizeof(T) == 4 || resident() == 0) return chunks;
    // a share's boundaries are rounded to planes, and it may start inside a column
    const long long cols = (long long)((p.n[0] + out_x - 1) / out_x) * ((p.n[1] + out_y - 1) / out_y);
    const long long even = cols * (3LL * p.n[2] + 2) / resident() + 1 + 2 + 2;
    return even < chunks.cost ? MhdPlan{0, even} : chunks;
  }
  static void launch(const PatchArgs<T>& a, const StageArgs& s, const MhdCoef<T>& mc, const sf_patch& p,
                     int mz, cudaStream_t st) {
    const dim3 block(MX, threads_y, 1);
    const dim3 grid((p.n[0] + out_x - 1) / out_x, (p.n[1] + out_y - 1) / out_y,
                    mz ? (p.n[2] + mz - 1) / mz : 1);
    if constexpr (ROWS == 0) {
      launch_after(kernel(), grid, block, smem, st, a, s, mc, mz);
    } else {
      const MhdWork wk = {mz, (int)grid.x, (int)grid.y};
      launch_after(kernel(), mz ? grid : dim3(resident()), block, smem, st, a, s, mc, wk);
    }
  }
};

// Without flux splitting: blocks of 15 or 7 output rows.  Both forms keep 16
// warps resident per SM (one block or two), so a plane of a round costs the
// same and the plans' costs compare; on a tie 15 rows, whose extra warp is 1
// in 16 instead of 1 in 8 (128^3 float: 1124 against 1155 us per step).
template <typename T, bool SPLIT, int VAR>
static void launch_instance(const PatchArgs<T>& a, const StageArgs& s, const MhdCoef<T>& mc,
                            const sf_patch& p, cudaStream_t st) {
  if constexpr (SPLIT) {
    using I = MhdInstance<T, VAR, 0>;
    I::launch(a, s, mc, p, I::plan(p).mz, st);
  } else {
    using A = MhdInstance<T, VAR, 15>;
    using B = MhdInstance<T, VAR, 7>;
    const MhdPlan pa = A::plan(p), pb = B::plan(p);
    if (pa.cost <= pb.cost)
      A::launch(a, s, mc, p, pa.mz, st);
    else
      B::launch(a, s, mc, p, pb.mz, st);
  }
}

template <typename T, bool SPLIT>
static void launch_variant(const PatchArgs<T>& a, const StageArgs& s, const MhdCoef<T>& mc,
                           const sf_patch& p, cudaStream_t st) {
  if (mc.variant == 1)
    launch_instance<T, SPLIT, 1>(a, s, mc, p, st);
  else if (mc.variant == 2)
    launch_instance<T, SPLIT, 2>(a, s, mc, p, st);
  else
    launch_instance<T, SPLIT, 0>(a, s, mc, p, st);
}

template <typename T>
static sf_status launch(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                        void* rhs_out, cudaStream_t st) {
  PatchArgs<T> a = make_args<T>(prm, p, stage, 8, rhs_out);
  const int last = prm.rk == SF_RK4 ? 3 : 2;
  if (p.cfl_rate && !rhs_out && stage == last) {
    if (cudaMemsetAsync(p.cfl_rate, 0, sizeof(double), st) != cudaSuccess)
      return set_error(SF_ECUDA, "reset of cfl_rate failed");
    a.rate = p.cfl_rate;
  }
  const MhdCoef<T> mc = coef<T>(prm, p);
  if (prm.flux_split)
    launch_variant<T, true>(a, s, mc, p, st);
  else
    launch_variant<T, false>(a, s, mc, p, st);
  return after_launch("mhd_stage_kernel");
}

sf_status launch_mhd(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                     void* rhs_out, cudaStream_t st) {
  if (p.precision == SF_FP64) return launch<double>(prm, p, s, stage, rhs_out, st);
  return launch<float>(prm, p, s, stage, rhs_out, st);
}

}  // namespace sf

using namespace sf;

extern "C" sf_status sf_mhd_max_rate(const sf_params* prm, const sf_patch* patch,
                                     const void* array, double* d_rate, void* stream) {
  if (!patch || !array || !d_rate) return set_error(SF_EINVAL, "NULL argument");
  sf_patch p = *patch;
  normalise_strides(p, 8);
  p.u_stage = const_cast<void*>(array);
  sf_status e = check_patch(prm, p, 0, 0);
  if (e) return e;
  if (p.system != SF_MHD) return set_error(SF_EINVAL, "sf_mhd_max_rate needs an SF_MHD patch");
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_rate, 0, sizeof(double), st) != cudaSuccess)
    return set_error(SF_ECUDA, "memset of d_rate failed");
  const long long total = (long long)p.n[0] * p.n[1] * p.n[2];
  int blocks = (int)((total + 255) / 256);
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (p.precision == SF_FP64)
    mhd_rate_kernel<double><<<blocks, 256, 0, st>>>((const double*)array, p.n[0], p.n[1], p.n[2],
                                                    p.ghost, p.sy, p.sz, p.sf, coef<double>(*prm, p),
                                                    (unsigned long long*)d_rate);
  else
    mhd_rate_kernel<float><<<blocks, 256, 0, st>>>((const float*)array, p.n[0], p.n[1], p.n[2],
                                                   p.ghost, p.sy, p.sz, p.sf, coef<float>(*prm, p),
                                                   (unsigned long long*)d_rate);
  return after_launch("mhd_rate_kernel");
}
