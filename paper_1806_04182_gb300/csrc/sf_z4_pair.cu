// The two-point CCZ4 stage kernel on the padded 96^3-class layout: 32 x 16 x 1
// tiles, compile-time strides (see sf_z4_pair.cuh).
#include "sf_z4_pair.cuh"

namespace sf {
namespace {

// The x ghost columns of every ghosted row (y and z over the whole ghosted
// range) of every field of u, from the same row's interior: ghost x = m
// (m < 3) takes x = m + n0, ghost x = n0 + 3 + m takes x = 3 + m.  Run after
// the stage kernel, whose fused y and z images have filled the interior part
// of the ghost rows.  One thread per ghost value.
__global__ void __launch_bounds__(256) pair_xghost_kernel(float* __restrict__ u, int nx, int ny,
                                                          int nz, long long sf) {
  const int Y = ny + 6, rows = Y * (nz + 6);
  const long long total = 25LL * rows * 6;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int q = (int)(t % 6);
    const long long row = t / 6;
    const int f = (int)(row / rows), r = (int)(row - (long long)f * rows);
    const int z = r / Y, y = r - z * Y;
    float* b = u + f * sf + (long long)z * kSZ + (long long)y * kSY;
    if (q < 3) b[q] = b[q + nx];
    else b[nx + q] = b[q];
  }
}

}  // namespace

template <typename H2, typename C, int FORM>
__global__ void __launch_bounds__(C::kThreads, 1)
    z4_pair_kernel(const __grid_constant__ CUtensorMap map, PatchArgs<float> a, StageArgs s,
                   Z4Coef<float> zc, const __grid_constant__ PairCoef pc,
                   const __grid_constant__ RkMaps rk) {
  extern __shared__ __align__(128) unsigned char smem[];
  // planes next to the z faces first (their tiles also write the z images, the
  // slowest tiles), so that the partial last wave holds plain tiles
  const int k = (int)((blockIdx.z + 3 * gridDim.z - 3) % gridDim.z);
  pair_tile<H2, C, FORM, false>(&map, rk.m, a, s, zc, &pc, blockIdx.x * 32, blockIdx.y * C::BY, k, smem);
}

namespace {

template <typename H2>
sf_status launch_pair(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                      void* rhs_out, cudaStream_t st) {
  using C = PairFlat;
  CUtensorMap map;
  if (sf_status e = encode_pair_map<C>(&map, p, p.u_stage, false)) return e;
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    for (auto f : {z4_pair_kernel<H2, C, kRkGeneric>, z4_pair_kernel<H2, C, kRk4First>,
                   z4_pair_kernel<H2, C, kRk4Mid>, z4_pair_kernel<H2, C, kRk4Last>})
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  });
  PatchArgs<float> a = make_args<float>(prm, p, stage, 25, rhs_out);
  const Z4Coef<float> zc = z4_coef<float>(prm);
  const PairCoef pc = pair_coef(prm, p);
  const int form = rk_form(s);
  RkMaps rk;
  if (sf_status e = encode_rk_maps<C>(&rk, p, form)) return e;
  const dim3 block(32, C::W, 1);
  const dim3 grid(p.n[0] / C::BX, p.n[1] / C::BY, p.n[2]);
  switch (form) {
    case kRk4First:
      launch_after(z4_pair_kernel<H2, C, kRk4First>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
      break;
    case kRk4Mid:
      launch_after(z4_pair_kernel<H2, C, kRk4Mid>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
      break;
    case kRk4Last:
      launch_after(z4_pair_kernel<H2, C, kRk4Last>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
      break;
    default:
      launch_after(z4_pair_kernel<H2, C, kRkGeneric>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
  }
  sf_status e = after_launch("z4_pair_kernel");
  // the RK4 forms write the x images themselves
  if (e || !s.ghosts || s.mode == 1 || form != kRkGeneric) return e;
  const long long total = 25LL * (p.n[1] + 6) * (p.n[2] + 6) * 6;
  const int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 8);
  pair_xghost_kernel<<<blocks, 256, 0, st>>>(a.nx, p.n[0], p.n[1], p.n[2], p.sf);
  return after_launch("pair_xghost_kernel");
}

}  // namespace

// The two-point kernel serves float storage with centred advection on the
// padded 96^3-class layout with the one-float row offset: 3 ghosts, row
// pitch 104 floats, plane pitch 104 x 102, field pitch a multiple of 4
// floats, every array 4 bytes past a 16-byte boundary, whole 32 x 16 tiles.
bool z4_pair_eligible(const sf_params& prm, const sf_patch& p, const void* rhs_out) {
  using C = PairFlat;
  if (p.system != SF_Z4 || p.precision == SF_FP64 || prm.lopsided) return false;
  if (p.ghost != 3 || p.sy != kSY || p.sz != kSZ || p.sf % 4) return false;
  if (p.n[0] % 32 || p.n[1] % C::BY || p.n[0] + 7 > kSY || p.n[1] + 6 > 102) return false;
  if (!offset_aligned(p.u_stage)) return false;
  if (rhs_out) return true;  // RHS output: scalar stores
  for (const void* q : {(const void*)p.u_n, (const void*)p.u_next, (const void*)p.acc})
    if (q && !offset_aligned(q)) return false;
  if (p.kahan && !offset_aligned(p.kahan)) return false;
  return true;
}

sf_status launch_z4_pair(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                         void* rhs_out, cudaStream_t st) {
  if (p.precision == SF_FP32_BULK_DW) return launch_pair<DW2>(prm, p, s, stage, rhs_out, st);
  return launch_pair<D2>(prm, p, s, stage, rhs_out, st);
}

}  // namespace sf
