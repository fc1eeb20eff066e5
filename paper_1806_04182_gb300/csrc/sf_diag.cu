// FP64 diagnostics of a patch: wave energy, CCZ4 constraint monitors
// (Theta, Z^i = chi/2 (Gammahat^i - Gamma~^i), ln det gt, tr A~; Sec. V) and a
// count of non-finite values.  Block partial sums are combined with double
// atomics into a 5-double device array that the caller owns.
#include "sf_internal.cuh"

namespace sf {

// A float's value as a double.  The conversion instruction runs at the FP64
// pipe's rate (17 cycles per warp and SM, an addition 20, predicated off as
// well); moving the bits takes some eight integer instructions, 2.4 cycles.
// Subnormals are not moved but reported in `sub` (EXACT: the instruction for
// every value).
template <bool EXACT>
__device__ __forceinline__ double dbl(float x, unsigned& sub) {
  if (EXACT) return (double)x;
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  sub |= m - 1u < 0x007fffffu ? 1u : 0u;
  // the exponent's bias, an exponent of all ones (inf, NaN) or zero
  const unsigned bias = m >= 0x7f800000u ? 0x70000000u : (m ? 0x38000000u : 0u);
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + bias)), (int)(m << 29));
}
template <bool EXACT>
__device__ __forceinline__ double dbl(double x, unsigned&) {
  return x;
}

__device__ __forceinline__ bool nonfinite(float x) { return (__float_as_uint(x) & 0x7f800000u) == 0x7f800000u; }
__device__ __forceinline__ bool nonfinite(double x) {
  return ((unsigned)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}

// ln d.  Near 1, where a conformal determinant stays, 2 atanh(z) with
// z = (d - 1)/(d + 1) by its series to z^13 (|z| < 1/32: the next term is below
// 2^-70 z); elsewhere log().
__device__ __forceinline__ double ln_near1(double d) {
  if (fabs(d - 1.0) >= 0.0625) return log(d);  // (NaN takes the series and stays NaN)
  const double z = (d - 1.0) / (d + 1.0), y = z * z;
  double p = fma(y, 2.0 / 13.0, 2.0 / 11.0);
  p = fma(y, p, 2.0 / 9.0);
  p = fma(y, p, 2.0 / 7.0);
  p = fma(y, p, 2.0 / 5.0);
  p = fma(y, p, 2.0 / 3.0);
  return fma(y * z, p, 2.0 * z);
}

// The CCZ4 monitors of one point: Theta^2, |Z|^2, (ln det)^2, (tr A~)^2; false
// if a subnormal value was met (float, not EXACT).  The kernel is bound by
// the FP64 pipe (87% busy), so the contractions are factored to the fewest
// operations, about 190 a point (with every Christoffel symbol formed apart and
// a conversion for each of the 89 values read, 96^3 float took 761 us; factored
// 468, values widened by integer instructions 344): with D_b g the unscaled
// derivative stencils and h_b = 1/(12 dx_b),
//   V_l = sum_b h_b sum_c ig^bc D_b g_lc - h_l/2 sum_bc ig^bc D_l g_bc,
//   Gamma~^a = sum_l ig^al V_l.
template <bool EXACT, typename T>
__device__ __forceinline__ bool z4_monitors(const T* __restrict__ p, long long F, long long sy,
                                            long long sz, const double (&ih)[3], double* m) {
  unsigned sub = 0u;
  auto at = [&](const T* q) { return dbl<EXACT>(*q, sub); };
  // float arrays hold chi, gt_ii and alpha minus 1 (flat-space offset)
  const double off = sizeof(T) == 4 ? 1.0 : 0.0;
  double gt[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) gt[q] = at(&p[(1 + q) * F]) + ((q == 0 || q == 3 || q == 5) ? off : 0.0);
  const double c00 = gt[3] * gt[5] - gt[4] * gt[4], c01 = gt[2] * gt[4] - gt[1] * gt[5],
               c02 = gt[1] * gt[4] - gt[2] * gt[3], c11 = gt[0] * gt[5] - gt[2] * gt[2],
               c12 = gt[1] * gt[2] - gt[0] * gt[4], c22 = gt[0] * gt[3] - gt[1] * gt[1];
  const double det = gt[0] * c00 + gt[1] * c01 + gt[2] * c02, idet = 1.0 / det;
  const double ig[6] = {c00 * idet, c01 * idet, c02 * idet, c11 * idet, c12 * idet, c22 * idet};
  constexpr int S[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
  double V[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const long long s = d == 0 ? 1 : (d == 1 ? sy : sz);
    double D[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const T* c = p + (1 + q) * F;
      D[q] = fma(8.0, at(&c[s]) - at(&c[-s]), at(&c[-2 * s]) - at(&c[2 * s]));
    }
    double od = ig[1] * D[1];
    od = fma(ig[2], D[2], od);
    od = fma(ig[4], D[4], od);
    double tr = ig[0] * D[0];
    tr = fma(ig[3], D[3], tr);
    tr = fma(ig[5], D[5], tr);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      double t = ig[S[d][0]] * D[S[l][0]];
      t = fma(ig[S[d][1]], D[S[l][1]], t);
      t = fma(ig[S[d][2]], D[S[l][2]], t);
      if (l == d) t -= fma(0.5, tr, od);
      V[l] = fma(ih[d], t, V[l]);
    }
  }
  double Z2 = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double z = at(&p[(14 + a) * F]);
#pragma unroll
    for (int l = 0; l < 3; ++l) z = fma(-ig[S[a][l]], V[l], z);
    Z2 = fma(z, z, Z2);
  }
  const double hchi = 0.5 * (at(&p[0]) + off);
  double trd = ig[0] * at(&p[8 * F]), tro = ig[1] * at(&p[9 * F]);
  trd = fma(ig[3], at(&p[11 * F]), trd);
  trd = fma(ig[5], at(&p[13 * F]), trd);
  tro = fma(ig[2], at(&p[10 * F]), tro);
  tro = fma(ig[4], at(&p[12 * F]), tro);
  const double trA = fma(2.0, tro, trd), Th = at(&p[17 * F]), ld = ln_near1(det);
  m[0] = Th * Th;
  m[1] = hchi * hchi * Z2;
  m[2] = ld * ld;
  m[3] = trA * trA;
  return sub == 0u;
}

// Three blocks per SM (at most 85 registers), which is also the grid: one round.
constexpr int kDiagBlocks = 3;
template <typename T, int SYSTEM>
__global__ void __launch_bounds__(256, kDiagBlocks) diag_kernel(const T* __restrict__ u0, int nx, int ny, int nz,
                                                   int g, long long sy, long long sz, long long F,
                                                   double hx, double hy, double hz, double* out) {
  const long long total = (long long)nx * ny * nz;
  constexpr int nf = SYSTEM == SF_WAVE ? 5 : (SYSTEM == SF_Z4 ? 25 : 8);
  double acc[4] = {0, 0, 0, 0};
  int bad = 0;
  const double ih[3] = {1.0 / (12.0 * hx), 1.0 / (12.0 * hy), 1.0 / (12.0 * hz)};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % nx);
    const int j = (int)((t / nx) % ny);
    const int k = (int)(t / ((long long)nx * ny));
    const T* p = u0 + (long long)(k + g) * sz + (long long)(j + g) * sy + (i + g);
#pragma unroll
    for (int f = 0; f < nf; ++f) bad += nonfinite(p[f * F]) ? 1 : 0;
    if (SYSTEM == SF_WAVE) {
      double e = 0.0;
      for (int f = 1; f < 5; ++f) {
        const double v = double(p[f * F]);
        e += 0.5 * v * v;
      }
      acc[0] += e * hx * hy * hz;
    } else if (SYSTEM == SF_Z4) {
      double m[4];
      if (!z4_monitors<false>(p, F, sy, sz, ih, m)) z4_monitors<true>(p, F, sy, sz, ih, m);
      for (int q = 0; q < 4; ++q) acc[q] += m[q];
    }
  }
  __shared__ double sm[5][256];
  for (int q = 0; q < 4; ++q) sm[q][threadIdx.x] = acc[q];
  sm[4][threadIdx.x] = (double)bad;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int q = 0; q < 5; ++q) sm[q][threadIdx.x] += sm[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 5; ++q) atomicAdd(out + q, sm[q][0]);
}

template <typename T>
static void launch_diag(const sf_patch& p, const void* array, double* out, int blocks, cudaStream_t st) {
  auto* kernel = p.system == SF_WAVE ? diag_kernel<T, SF_WAVE>
                                     : (p.system == SF_Z4 ? diag_kernel<T, SF_Z4> : diag_kernel<T, SF_MHD>);
  kernel<<<blocks, 256, 0, st>>>((const T*)array, p.n[0], p.n[1], p.n[2], p.ghost, p.sy, p.sz, p.sf,
                                 p.dx[0], p.dx[1], p.dx[2], out);
}

}  // namespace sf

using namespace sf;

extern "C" sf_status sf_diagnostics(const sf_params* prm, const sf_patch* patch, const void* array,
                                    double* d_out, void* stream) {
  if (!patch || !array || !d_out) return set_error(SF_EINVAL, "NULL argument");
  sf_patch p = *patch;
  normalise_strides(p, sf_nfields(p.system));
  p.u_stage = const_cast<void*>(array);
  sf_status e = check_patch(prm, p, 0, 0);
  if (e) return e;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_out, 0, 5 * sizeof(double), st) != cudaSuccess)
    return set_error(SF_ECUDA, "memset of d_out failed");
  const long long total = (long long)p.n[0] * p.n[1] * p.n[2];
  int blocks = (int)((total + 255) / 256);
  if (blocks > 152 * kDiagBlocks) blocks = 152 * kDiagBlocks;
  if (p.precision == SF_FP64)
    launch_diag<double>(p, array, d_out, blocks, st);
  else
    launch_diag<float>(p, array, d_out, blocks, st);
  return after_launch("diag_kernel");
}
