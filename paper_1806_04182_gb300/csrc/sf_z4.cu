// Standalone CCZ4 stage kernel (one launch per patch); the per-point
// right-hand side lives in sf_z4.cuh.  Float storage with centred advection
// and row / plane / field pitches on 16-byte boundaries goes to the
// TMA-staged kernels (sf_z4_tma.cu).  Layouts with the
// strides of a dense 96^3 patch with 3 ghosts get a kernel with compile-time
// strides; every other layout, and one-sided advection, uses runtime strides.
#include <algorithm>

#include "sf_internal.cuh"
#include "sf_z4.cuh"

namespace sf {

// 128 threads and at least MINB CTAs per SM.  float: 3 (<= 168 registers): on
// the 96^3 benchmark patch this measured faster than 2 CTAs (255 registers)
// and than 4+ CTAs (128 registers or fewer, with spills).  double is bound by
// the FP64 pipe (2435 operations a point; 87% busy at 2 CTAs): 3 CTAs spill
// but leave the pipe less idle between loads and writes (96^3 step 15.99 ->
// 15.90 ms, 61 x 47 x 53 3.28 -> 3.10 ms, with one-sided advection 4.38 -> 4.04
// ms), except where an SM's share of the patch is 1, 2 or 4 CTAs: up to 2 the
// spills only lengthen the one round (20^3 395 against 406 us, 32^3 730 against
// 735 us), and 3 + 1 leaves the last CTA alone where 2 + 2 does not (37 x 55 x
// 19 one-sided 2.19 against 1.84 ms).  In z4_rhs's order of operations (2820 a point) the
// 96^3 step took 18.65 ms.
//
// The right-hand sides of the 25 fields are parked in shared memory as
// z4_cell produces them, and the RK stage combination (which reads U^n, the
// accumulator and the Kahan term from memory) runs once at the end as a
// rolled loop over the fields.  Inlined after every field, the combination
// put 25 copies of its code and 25 dependent DRAM reads into the middle of the
// computation; the deferred form measured 7-10% faster on the 96^3 patch.
template <typename T, typename H, int SY, int SZ, bool LOP, int MINB>
__global__ void __launch_bounds__(128, MINB)
    z4_stage_kernel(PatchArgs<T> a, StageArgs s, Z4Coef<T> zc) {
  __shared__ T rbuf[25 * 128];
  wait_predecessor();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= a.n[0] || j >= a.n[1]) return;
  const int g = a.g;
  const long long sy = SY ? (long long)SY : a.sy;
  const long long sz = SZ ? (long long)SZ : a.sz;
  const long long c = (long long)(k + g) * sz + (long long)(j + g) * sy + (i + g);
  GlobalSrc<T, SY, SZ, LOP> src{a.us + c, a.sf, a.sy, a.sz};
  const Images im = ghost_images(a, s, i, j, k);
  const int tid = threadIdx.y * 32 + threadIdx.x;
  z4_cell<T, H, LOP>(a, zc, src, [&](int f, T r, T) { rbuf[f * 128 + tid] = r; });
  write_fields<T, 25>(a, s, im, c, i, j, k, rbuf + tid, 128);
}

template <typename T, typename H, int MINB>
static void launch_kernel(const PatchArgs<T>& a, const StageArgs& s, const sf_params& prm, const sf_patch& p,
                          dim3 grid, cudaStream_t st) {
  const Z4Coef<T> zc = z4_coef<T>(prm);
  const dim3 block(32, 4, 1);
  if (prm.lopsided)
    launch_after(z4_stage_kernel<T, H, 0, 0, true, MINB>, grid, block, 0, st, a, s, zc);
  else if (p.sy == 102 && p.sz == 102 * 102)
    launch_after(z4_stage_kernel<T, H, 102, 102 * 102, false, MINB>, grid, block, 0, st, a, s, zc);
  else
    launch_after(z4_stage_kernel<T, H, 0, 0, false, MINB>, grid, block, 0, st, a, s, zc);
}

template <typename T, typename H>
static sf_status launch(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                        void* rhs_out, cudaStream_t st) {
  const PatchArgs<T> a = make_args<T>(prm, p, stage, 25, rhs_out);
  const dim3 grid((p.n[0] + 31) / 32, (p.n[1] + 3) / 4, p.n[2]);
  if constexpr (sizeof(T) == 8) {
    const long long sms = std::max(1, sm_count());
    const long long share = ((long long)grid.x * grid.y * grid.z + sms - 1) / sms;
    if (share <= 2 || share == 4) {
      launch_kernel<T, H, 2>(a, s, prm, p, grid, st);
      return after_launch("z4_stage_kernel");
    }
  }
  launch_kernel<T, H, 3>(a, s, prm, p, grid, st);
  return after_launch("z4_stage_kernel");
}

sf_status launch_z4(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                    void* rhs_out, cudaStream_t st) {
  if (z4_pair_eligible(prm, p, rhs_out)) return launch_z4_pair(prm, p, s, stage, rhs_out, st);
  if (z4_pair_any_eligible(prm, p, s, rhs_out)) return launch_z4_pair_any(prm, p, s, stage, st);
  if (z4_tma_any_eligible(prm, p)) return launch_z4_tma(prm, p, s, stage, rhs_out, st);
  if (p.precision == SF_FP64) return launch<double, double>(prm, p, s, stage, rhs_out, st);
  if (p.precision == SF_FP32_BULK_DW) return launch<float, dw>(prm, p, s, stage, rhs_out, st);
  return launch<float, double>(prm, p, s, stage, rhs_out, st);
}

}  // namespace sf
