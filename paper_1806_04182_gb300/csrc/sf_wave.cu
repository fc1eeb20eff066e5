// Standalone wave stage kernel (one launch per patch), forward or adjoint;
// the per-point right-hand side lives in sf_wave.cuh.
#include "sf_internal.cuh"
#include "sf_wave.cuh"

namespace sf {

template <typename T, bool ADJ>
__global__ void __launch_bounds__(128, 4) wave_stage_kernel(PatchArgs<T> a, StageArgs s) {
  wait_predecessor();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= a.n[0] || j >= a.n[1]) return;
  if (s.mode == 1) {
    const int g = a.g;
    T v[5], r[5];
    wave_point<T, ADJ>(a, a.us + (long long)(k + g) * a.sz + (long long)(j + g) * a.sy + (i + g), v, r);
#pragma unroll
    for (int f = 0; f < 5; ++f) a.nx[f * a.ninterior + ((long long)k * a.n[1] + j) * a.n[0] + i] = r[f];
    return;
  }
  wave_stage_point<T, ADJ>(a, s, i, j, k);
}

// float: a block of 32 x 8 columns marches mz planes in z.  Planes of the
// stage input come into a ring of shared memory slots (cp.async, with the halo
// of 3 in x and y, two planes ahead), so each value of a plane is read from L2
// about 2.1 times instead of 19 times from L1; x and y neighbours come from
// the plane's slot, z neighbours from a register window of the thread's own
// column, and the RK inputs of the next plane are read ahead.  One barrier per
// plane: it makes the plane that enters the window visible and frees the slot
// of the plane before.  Bound by the latency of those reads at 24 warps per
// SM (HBM would take 31 us): 128^3 RK4 stage 97 us with one point per thread
// and every stencil read from global memory, 62 us now; 32 x 16 columns one
// block per SM 78 us, 32 x 8 two per SM 67 us, without the read-ahead 65 us.
// The arithmetic is that of wave_stage_kernel, bit for bit.
constexpr int kMarchX = 32, kMarchY = 8, kMarchCols = kMarchX + 6, kMarchCells = kMarchCols * (kMarchY + 6);
constexpr int kMarchSlots = 6;
constexpr int kMarchSmem = kMarchSlots * 5 * kMarchCells * 4;

// The periodic images of a point's five new values (store_images, each image's
// offset formed once for the fields).
__device__ __forceinline__ void store_images5(const PatchArgs<float>& a, unsigned m, int c, int sf,
                                              const float* q) {
  const int dz = a.n[2] * (int)a.sz, dy = a.n[1] * (int)a.sy, dx = a.n[0];
#pragma unroll 1
  for (int p = 0; p < 3; ++p) {
    if (p && !(m >> (3 + p) & 1u)) continue;
    const int oz = p == 0 ? 0 : (p == 1 ? dz : -dz);
#pragma unroll 1
    for (int u = 0; u < 3; ++u) {
      if (u && !(m >> (1 + u) & 1u)) continue;
      const int oy = oz + (u == 0 ? 0 : (u == 1 ? dy : -dy));
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        if ((w && !(m >> (w - 1) & 1u)) || !(p | u | w)) continue;
        float* o = a.nx + (c + oy + (w == 0 ? 0 : (w == 1 ? dx : -dx)));
#pragma unroll
        for (int f = 0; f < 5; ++f, o += sf) *o = q[f];
      }
    }
  }
}

// FORM: the RK4 stage with the compensated accumulator, fixed at compile time
// (0: stage 0 with U^n the stage input, 1: stages 1 and 2, 2: stage 3).  All
// element offsets fit 32 bits (march_planes).
template <bool ADJ, int FORM>
__global__ void __launch_bounds__(kMarchX * kMarchY, 3)
    wave_march_kernel(PatchArgs<float> a, StageArgs s, int mz) {
  extern __shared__ __align__(16) float ring[];  // [slot][field][cell]
  constexpr int NC = kMarchCells, CW = kMarchCols, NT = kMarchX * kMarchY, NS = (NC + NT - 1) / NT;
  constexpr int SLOT = 5 * NC, RING = kMarchSlots * SLOT;
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * kMarchX + tx;
  const int x0 = blockIdx.x * kMarchX, y0 = blockIdx.y * kMarchY;
  const int i = x0 + tx, j = y0 + ty, g = a.g;
  const int sy = (int)a.sy, sz = (int)a.sz, sf = (int)a.sf;
  const int k0 = blockIdx.z * mz, k1 = min(k0 + mz, a.n[2]);
  const bool out = i < a.n[0] && j < a.n[1];
  // columns outside the patch repeat the last one; their results go nowhere
  int c = (k0 + g) * sz + (min(j, a.n[1] - 1) + g) * sy + (min(i, a.n[0] - 1) + g);
  int so[NS];
#pragma unroll
  for (int e = 0; e < NS; ++e) {
    const int t = tid + e * NT;
    const int cx = min(x0 - 3 + t % CW, a.n[0] + 2), cy = min(y0 - 3 + t / CW, a.n[1] + 2);
    so[e] = (k0 + g) * sz + (cy + g) * sy + (cx + g);
  }
  wait_predecessor();
  const unsigned ring0 = (unsigned)__cvta_generic_to_shared(ring) + tid * 4;
  int left = k1 + 3 - k0;  // planes still to be staged
  int ws = 0;              // slot they go to, in elements
  auto stage = [&]() {  // the next plane into its slot, one group
    if (left-- > 0) {
#pragma unroll
      for (int e = 0; e < NS; ++e) {
        if ((e + 1) * NT <= NC || tid + e * NT < NC) {
#pragma unroll
          for (int f = 0; f < 5; ++f)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                             ring0 + 4u * (ws + f * NC + e * NT)),
                         "l"(a.us + (so[e] + f * sf))
                         : "memory");
        }
        so[e] += sz;
      }
      ws = ws + SLOT == RING ? 0 : ws + SLOT;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int p = 0; p < 5; ++p) stage();
  float w[5][7];  // planes k - 3 .. k + 3 of the thread's column
#pragma unroll
  for (int f = 0; f < 5; ++f)
#pragma unroll
    for (int q = 1; q < 4; ++q) w[f][q] = a.us[c + f * sf + (q - 4) * sz];
  const float* lc = ring + (ty + 3) * CW + tx + 3;
  // planes k0 .. k0 + 2 have landed
  asm volatile("cp.async.wait_group 2;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int f = 0; f < 5; ++f)
#pragma unroll
    for (int q = 0; q < 3; ++q) w[f][4 + q] = lc[q * SLOT + f * NC];
  int ps = 0, ns = 3 * SLOT;  // slots of planes k and k + 3
  const unsigned xy = ghost_images(a, s, i, j, 0).mask & 15u;
  float un2[5], acc2[5];  // the next plane's U^n and accumulator
  auto rk_in = [&](int o) {
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      if (FORM > 0) un2[f] = a.un[o + f * sf];
      if (FORM > 0) acc2[f] = a.acc[o + f * sf];
    }
  };
  rk_in(c);
  float bad = 0.0f;  // any non-finite output makes it NaN
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();  // plane k + 3 visible; plane k - 1's slot is free
    stage();
    float un[5], acc[5], kh[5], v[5], r[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      if (FORM > 0) un[f] = un2[f];
      if (FORM > 0) acc[f] = acc2[f];
      if (FORM > 1) kh[f] = a.kh[c + f * sf];
    }
    if (k + 1 < k1) rk_in(c + sz);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
#pragma unroll
      for (int q = 0; q < 6; ++q) w[f][q] = w[f][q + 1];
      w[f][6] = lc[ns + f * NC];
      v[f] = w[f][3];
    }
    const float* pl = lc + ps;
    wave_rhs<float, ADJ>(
        a, [&](int f, int d, int o) { return d == 2 ? w[f][3 + o] : pl[f * NC + o * (d == 0 ? 1 : CW)]; }, v, r);
    if (out) {
      float q[5];
#pragma unroll
      for (int f = 0; f < 5; ++f) {  // stage_combine of the form
        const int o = c + f * sf;
        if (FORM == 0) {
          a.acc[o] = 0.0f + a.c_acc * r[f];
          q[f] = v[f] + a.c_next * r[f];
        } else if (FORM == 1) {
          a.acc[o] = acc[f] + a.c_acc * r[f];
          q[f] = un[f] + a.c_next * r[f];
        } else {
          const float inc = acc[f] + a.c_next * r[f];
          const float y = inc - kh[f];
          q[f] = un[f] + y;
          a.kh[o] = (q[f] - un[f]) - y;
        }
        a.nx[o] = q[f];
        bad += q[f] * 0.0f;
      }
      Images im;
      im.mask = s.ghosts ? xy | (k < g ? 16u : 0u) | (k >= a.n[2] - g ? 32u : 0u) : 0u;
      if (im.mask) store_images5(a, im.mask, c, sf, q);
    }
    c += sz;
    ps = ps + SLOT == RING ? 0 : ps + SLOT;
    ns = ns + SLOT == RING ? 0 : ns + SLOT;
  }
  if (s.check_finite && bad != bad) atomicOr(s.status, ST_NONFINITE);
}

// Planes per block of the marching kernel for a patch, 0 where it does not
// serve.  It needs enough points to hide its serial planes (RK4 step, against
// one point per thread: 48^3 57 against 41 us, 64^3 59 against 64, 96^3 114
// against 154, 128^3 248 against 388), and element offsets of 32 bits.  A
// block's cost is its planes plus about 4 planes' time to start (the ring's
// first loads and the window), in
// rounds of the resident blocks.
constexpr long long kMarchPoints = 200000;
static int march_planes(const sf_patch& p) {
  static int resident[64] = {0};
  if (5 * p.sf >= (1LL << 31) || (long long)p.n[0] * p.n[1] * p.n[2] < kMarchPoints) return 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!resident[dev]) {
    int per_sm = 0, sms = 0;
    for (auto f : {wave_march_kernel<false, 0>, wave_march_kernel<false, 1>, wave_march_kernel<false, 2>,
                   wave_march_kernel<true, 0>, wave_march_kernel<true, 1>, wave_march_kernel<true, 2>})
      if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMarchSmem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, wave_march_kernel<false, 2>, kMarchX * kMarchY,
                                                      kMarchSmem) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    resident[dev] = per_sm * sms;
  }
  const long long cols = (long long)((p.n[0] + kMarchX - 1) / kMarchX) * ((p.n[1] + kMarchY - 1) / kMarchY);
  int best = 0;
  long long cost = -1;
  for (int mz = 64; mz >= 1; --mz) {
    if ((p.n[2] + mz - 1) / mz > 65535) break;
    const long long blocks = cols * ((p.n[2] + mz - 1) / mz);
    const long long t = (blocks + resident[dev] - 1) / resident[dev] * (mz + 4);
    if (cost < 0 || t < cost) {
      cost = t;
      best = mz;
    }
  }
  return best;
}

template <typename T>
static sf_status launch(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                        void* rhs_out, bool adj, cudaStream_t st) {
  PatchArgs<T> a = make_args<T>(prm, p, stage, 5, rhs_out);
  if constexpr (sizeof(T) == 4) {
    const int form = s.mode != 0 || s.rk != SF_RK4 || !s.kahan || (stage == 0) != (s.un_alias != 0)
                         ? -1
                         : (stage == 0 ? 0 : (stage < 3 ? 1 : 2));
    const int mz = form >= 0 ? march_planes(p) : 0;
    if (mz > 0) {
      const dim3 grid((p.n[0] + kMarchX - 1) / kMarchX, (p.n[1] + kMarchY - 1) / kMarchY, (p.n[2] + mz - 1) / mz);
      auto* kernel = adj ? (form == 0 ? wave_march_kernel<true, 0>
                                      : (form == 1 ? wave_march_kernel<true, 1> : wave_march_kernel<true, 2>))
                         : (form == 0 ? wave_march_kernel<false, 0>
                                      : (form == 1 ? wave_march_kernel<false, 1> : wave_march_kernel<false, 2>));
      launch_after(kernel, grid, dim3(kMarchX, kMarchY), kMarchSmem, st, a, s, mz);
      return after_launch("wave_march_kernel");
    }
  }
  dim3 block(32, 4, 1);
  dim3 grid((p.n[0] + 31) / 32, (p.n[1] + 3) / 4, p.n[2]);
  launch_after(adj ? wave_stage_kernel<T, true> : wave_stage_kernel<T, false>, grid, block, 0, st, a, s);
  return after_launch("wave_stage_kernel");
}

sf_status launch_wave(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                      void* rhs_out, bool adjoint, cudaStream_t st) {
  if (p.precision == SF_FP64) return launch<double>(prm, p, s, stage, rhs_out, adjoint, st);
  return launch<float>(prm, p, s, stage, rhs_out, adjoint, st);
}

}  // namespace sf
