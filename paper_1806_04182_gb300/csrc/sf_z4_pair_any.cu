// The two-point CCZ4 tile (sf_z4_pair.cuh) for patches of any size on the
// one-float row offset layout: runtime strides, tiles that overhang the patch
// with masked stores, one patch per launch or the tiles of many patches.
//
// Two tile shapes of 512 points, 32 x 8 x 2 and 16 x 8 x 4; a patch takes the one
// that covers it with fewer tiles (kPairShapes; the wide one on a tie).  Lanes
// outside the patch idle: with 32 x 16 x 1 tiles alone, 36% of them on patches
// of 16 to 64 points a side and 25% on 48^3, with the two shapes 23% and none
// (96 mixed patches 11.6 -> 10.0 ms per RK4 step, eight 48^3 patches with halo
// exchange 1.59 -> 1.36 ms; a multi-plane tile by itself costs some 15% more
// than a flat one, so the padded 96^3-class layout keeps those).
#include "sf_z4_pair.cuh"

namespace sf {

// 8 slots each (9, 7 and 5: 3%, 1% and 4% slower on eight 48^3 patches)
using PairWide = PairShape<32, 8, 2, 8, 9>;
using PairDeep = PairShape<16, 8, 4, 8, 9>;

int z4_pair_shape(const sf_patch& p) {
  auto tiles = [&](const int* t) {
    long long n = 1;
    for (int d = 0; d < 3; ++d) n *= (p.n[d] + t[d] - 1) / t[d];
    return n;
  };
  return tiles(kPairShapes[1]) < tiles(kPairShapes[0]) ? 1 : 0;
}

// One CTA per tile of one patch (the RK4 Kahan forms).
template <typename C, int FORM>
__global__ void __launch_bounds__(C::kThreads, 1)
    z4_pair_any_kernel(const __grid_constant__ CUtensorMap map, PatchArgs<float> a, StageArgs s,
                       Z4Coef<float> zc, const __grid_constant__ PairCoef pc,
                       const __grid_constant__ RkMaps rk) {
  extern __shared__ __align__(128) unsigned char smem[];
  // the planes next to the z faces first, as in z4_pair_kernel
  const int z = (int)((blockIdx.z + 3 * gridDim.z - 3) % gridDim.z);
  pair_tile<DW2, C, FORM, true>(&map, rk.m, a, s, zc, &pc, blockIdx.x * C::BX, blockIdx.y * C::BY,
                                z * C::BZ, smem);
}

// The same over the tiles of many patches (the float CCZ4 patches of a batch
// on the two-point layout): one CTA per tile, the first n0 of the wide shape,
// the rest of the deep one; the tile's patch from `tl`, its stage arguments
// and stencil weights copied into shared memory, its tensor maps from `maps`
// (six per patch: RK chunks of U^n, accumulator and Kahan term, then the
// stencil boxes of the u_n, u_stage and u_next buffer roles; `role` picks the
// stage input).
template <int FORM>
__global__ void __launch_bounds__(32 * kPairWarps, 1)
    z4_pair_batch_kernel(const CUtensorMap* __restrict__ maps, int role,
                         const PatchArgs<float>* __restrict__ args, const PairCoef* __restrict__ coefs,
                         const TmaTile* __restrict__ tl, int n0, StageArgs s, Z4Coef<float> zc) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ PatchArgs<float> pa;
  __shared__ PairCoef pcs;
  wait_predecessor();
  const TmaTile w = tl[blockIdx.x];
  {
    static_assert(sizeof(PatchArgs<float>) % 4 == 0 && sizeof(PairCoef) % 4 == 0, "word copy");
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int* from = reinterpret_cast<const int*>(args + w.patch);
    int* to = reinterpret_cast<int*>(&pa);
    for (int q = tid; q < (int)(sizeof(PatchArgs<float>) / 4); q += 32 * kPairWarps) to[q] = from[q];
    from = reinterpret_cast<const int*>(coefs + w.patch);
    to = reinterpret_cast<int*>(&pcs);
    for (int q = tid; q < (int)(sizeof(PairCoef) / 4); q += 32 * kPairWarps) to[q] = from[q];
  }
  // (pair_tile's first barrier orders these copies before their reads)
  const CUtensorMap* pm = maps + 6 * (size_t)w.patch;
  if ((int)blockIdx.x < n0)
    pair_tile<DW2, PairWide, FORM, true>(pm + 3 + role, pm, pa, s, zc, &pcs, w.x0, w.y0, w.z0, smem);
  else
    pair_tile<DW2, PairDeep, FORM, true>(pm + 3 + role, pm, pa, s, zc, &pcs, w.x0, w.y0, w.z0, smem);
}

namespace {

template <typename C>
sf_status launch_any(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                     cudaStream_t st) {
  CUtensorMap map;
  if (sf_status e = encode_pair_map<C>(&map, p, p.u_stage, false)) return e;
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    for (auto f : {z4_pair_any_kernel<C, kRk4First>, z4_pair_any_kernel<C, kRk4Mid>, z4_pair_any_kernel<C, kRk4Last>})
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  });
  const PatchArgs<float> a = make_args<float>(prm, p, stage, 25, nullptr);
  const Z4Coef<float> zc = z4_coef<float>(prm);
  const PairCoef pc = pair_coef(prm, p);
  const int form = rk_form(s);
  RkMaps rk;
  if (sf_status e = encode_rk_maps<C>(&rk, p, form)) return e;
  const dim3 block(32, C::W, 1);
  const dim3 grid((p.n[0] + C::BX - 1) / C::BX, (p.n[1] + C::BY - 1) / C::BY, (p.n[2] + C::BZ - 1) / C::BZ);
  switch (form) {
    case kRk4First:
      launch_after(z4_pair_any_kernel<C, kRk4First>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
      break;
    case kRk4Mid:
      launch_after(z4_pair_any_kernel<C, kRk4Mid>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
      break;
    default:
      launch_after(z4_pair_any_kernel<C, kRk4Last>, grid, block, C::kSmemBytes, st, map, a, s, zc, pc, rk);
  }
  return after_launch("z4_pair_any_kernel");
}

template <typename C>
sf_status encode_batch(void* maps6, const sf_patch& p) {
  const void* arr[6] = {p.u_n, p.acc, p.kahan, p.u_n, p.u_stage, p.u_next};
  for (int q = 0; q < 6; ++q) {
    CUtensorMap m;
    if (sf_status e = encode_pair_map<C>(&m, p, arr[q], q < 3)) return e;
    memcpy(static_cast<char*>(maps6) + q * sizeof(CUtensorMap), &m, sizeof(m));
  }
  return SF_OK;
}

}  // namespace

// Any size on the one-float row offset layout: double-word islands, the RK4
// Kahan stage forms, pitches of a multiple of 4 floats with room for the
// float before each row, every array 4 bytes past a 16-byte boundary.
bool z4_pair_any_eligible(const sf_params& prm, const sf_patch& p, const StageArgs& s,
                          const void* rhs_out) {
  if (rhs_out || rk_form(s) == kRkGeneric) return false;
  return z4_pair_batch_eligible(prm, p);
}

sf_status launch_z4_pair_any(const sf_params& prm, const sf_patch& p, const StageArgs& s, int stage,
                             cudaStream_t st) {
  if (z4_pair_shape(p)) return launch_any<PairDeep>(prm, p, s, stage, st);
  return launch_any<PairWide>(prm, p, s, stage, st);
}

// Batch form: float CCZ4 with double-word islands, centred advection, 3
// ghosts, row / plane / field pitches of a multiple of 4 floats with room for
// the float before each row (row pitch >= n0 + 7), every array 4 bytes past
// a 16-byte boundary; any interior size (tiles may overhang).
bool z4_pair_batch_eligible(const sf_params& prm, const sf_patch& p) {
  if (p.system != SF_Z4 || p.precision != SF_FP32_BULK_DW || prm.lopsided) return false;
  if (p.ghost != 3 || p.sy % 4 || p.sz % 4 || p.sf % 4 || p.sy < p.n[0] + 7) return false;
  for (const void* q : {(const void*)p.u_n, (const void*)p.u_stage, (const void*)p.u_next,
                        (const void*)p.acc, (const void*)p.kahan})
    if (!offset_aligned(q)) return false;
  return true;
}

size_t z4_pair_coef_bytes() { return sizeof(PairCoef); }

// The six tensor maps of a batch patch (RK chunks of u_n, acc, kahan; stencil
// boxes of u_n, u_stage, u_next) for its tile shape, and its stencil weights.
sf_status encode_z4_pair_batch(void* maps6, void* coef, const sf_params& prm, const sf_patch& p) {
  if (sf_status e = z4_pair_shape(p) ? encode_batch<PairDeep>(maps6, p) : encode_batch<PairWide>(maps6, p))
    return e;
  const PairCoef pc = pair_coef(prm, p);
  memcpy(coef, &pc, sizeof(pc));
  return SF_OK;
}

sf_status launch_z4_pair_batch(const sf_params& prm, const void* d_maps, int role,
                               const PatchArgs<float>* d_args, const void* d_coefs,
                               const TmaTile* d_tiles, int ntiles, int nwide, const StageArgs& s,
                               cudaStream_t st) {
  if (ntiles <= 0) return SF_OK;
  constexpr int smem =
      PairWide::kSmemBytes > PairDeep::kSmemBytes ? PairWide::kSmemBytes : PairDeep::kSmemBytes;
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    for (auto f : {z4_pair_batch_kernel<kRk4First>, z4_pair_batch_kernel<kRk4Mid>, z4_pair_batch_kernel<kRk4Last>})
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  });
  const Z4Coef<float> zc = z4_coef<float>(prm);
  const CUtensorMap* maps = static_cast<const CUtensorMap*>(d_maps);
  const PairCoef* coefs = static_cast<const PairCoef*>(d_coefs);
  const dim3 block(32, kPairWarps, 1);
  switch (rk_form(s)) {
    case kRk4First:
      launch_after(z4_pair_batch_kernel<kRk4First>, ntiles, block, smem, st, maps, role, d_args, coefs, d_tiles, nwide, s, zc);
      break;
    case kRk4Mid:
      launch_after(z4_pair_batch_kernel<kRk4Mid>, ntiles, block, smem, st, maps, role, d_args, coefs, d_tiles, nwide, s, zc);
      break;
    case kRk4Last:
      launch_after(z4_pair_batch_kernel<kRk4Last>, ntiles, block, smem, st, maps, role, d_args, coefs, d_tiles, nwide, s, zc);
      break;
    default:
      return set_error(SF_EINVAL, "batched two-point tiles need the RK4 Kahan forms");
  }
  return after_launch("z4_pair_batch_kernel");
}

}  // namespace sf
