// The two-point CCZ4 tile (sf_z4_pair.cuh) over the tiles of many patches of any
// size, in one launch: all in one shape (kPairShapes) and that shape's kernel,
// or, where that saves rounds, each in the wide or the deep one, in a kernel
// that holds both tile bodies (z4_pair_batch_shapes).  (A kernel with all three
// spills: 96 mixed patches 9.96 instead of 9.52 ms, eight 48^3 patches 1.41
// instead of 1.36.)
#include <algorithm>
#include <type_traits>

#include "sf_z4_pair.cuh"

namespace sf {

// Tiles of many patches (the float CCZ4 patches of a batch
// on the two-point layout): one CTA per tile, the first n0 of shape C0, the
// rest of C1; the tile's patch from `tl`, its stage arguments
// and stencil weights copied into shared memory, its tensor maps from `maps`
// (six per patch: RK chunks of U^n, accumulator and Kahan term, then the
// stencil boxes of the u_n, u_stage and u_next buffer roles; `role` picks the
// stage input).
template <typename C0, typename C1, int FORM>
__global__ void __launch_bounds__(32 * kPairWarps, 1)
    z4_pair_batch_kernel(const CUtensorMap* __restrict__ maps, int role,
                         const PatchArgs<float>* __restrict__ args, const PairCoef* __restrict__ coefs,
                         const TmaTile* __restrict__ tl, int n0, StageArgs s,
                         Z4Coef<float> zc) {
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
  if constexpr (!std::is_same<C0, C1>::value) {
    if ((int)blockIdx.x >= n0) {
      pair_tile<DW2, C1, FORM, true>(pm + 3 + role, pm, pa, s, zc, &pcs, w.x0, w.y0, w.z0, smem);
      return;
    }
  }
  pair_tile<DW2, C0, FORM, true>(pm + 3 + role, pm, pa, s, zc, &pcs, w.x0, w.y0, w.z0, smem);
}

namespace {

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

template <typename C0, typename C1>
sf_status launch_shapes(const sf_params& prm, const void* d_maps, int role, const PatchArgs<float>* d_args,
                        const void* d_coefs, const TmaTile* d_tiles, int ntiles, int n0,
                        const StageArgs& s, cudaStream_t st) {
  constexpr int smem = std::max(C0::kSmemBytes, C1::kSmemBytes);
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    for (auto f : {z4_pair_batch_kernel<C0, C1, kRk4First>, z4_pair_batch_kernel<C0, C1, kRk4Mid>,
                   z4_pair_batch_kernel<C0, C1, kRk4Last>})
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  });
  const Z4Coef<float> zc = z4_coef<float>(prm);
  const CUtensorMap* maps = static_cast<const CUtensorMap*>(d_maps);
  const PairCoef* coefs = static_cast<const PairCoef*>(d_coefs);
  auto* kernel = z4_pair_batch_kernel<C0, C1, kRk4First>;
  switch (rk_form(s)) {
    case kRk4First: break;
    case kRk4Mid: kernel = z4_pair_batch_kernel<C0, C1, kRk4Mid>; break;
    case kRk4Last: kernel = z4_pair_batch_kernel<C0, C1, kRk4Last>; break;
    default: return set_error(SF_EINVAL, "batched two-point tiles need the RK4 Kahan forms");
  }
  launch_after(kernel, ntiles, dim3(32, kPairWarps, 1), smem, st, maps, role, d_args, coefs, d_tiles, n0, s, zc);
  return after_launch("z4_pair_batch_kernel");
}

}  // namespace

size_t z4_pair_coef_bytes() { return sizeof(PairCoef); }

// The six tensor maps of a batch patch (RK chunks of u_n, acc, kahan; stencil
// boxes of u_n, u_stage, u_next) for tile shape w, and its stencil weights.
sf_status encode_z4_pair_batch(void* maps6, void* coef, const sf_params& prm, const sf_patch& p, int w) {
  if (sf_status e = w == 0 ? encode_batch<PairFlat>(maps6, p)
                           : (w == 1 ? encode_batch<PairWide>(maps6, p) : encode_batch<PairDeep>(maps6, p)))
    return e;
  const PairCoef pc = pair_coef(prm, p);
  memcpy(coef, &pc, sizeof(pc));
  return SF_OK;
}

sf_status launch_z4_pair_batch(const sf_params& prm, const void* d_maps, int role,
                               const PatchArgs<float>* d_args, const void* d_coefs,
                               const TmaTile* d_tiles, const int* ends, const StageArgs& s,
                               cudaStream_t st) {
  const int n = ends[2];
  if (n <= 0) return SF_OK;
  if (ends[0] == n)
    return launch_shapes<PairFlat, PairFlat>(prm, d_maps, role, d_args, d_coefs, d_tiles, n, n, s, st);
  if (ends[0] != 0) return set_error(SF_EINVAL, "flat two-point tiles beside others");
  if (ends[1] == n)
    return launch_shapes<PairWide, PairWide>(prm, d_maps, role, d_args, d_coefs, d_tiles, n, n, s, st);
  if (ends[1] == 0)
    return launch_shapes<PairDeep, PairDeep>(prm, d_maps, role, d_args, d_coefs, d_tiles, n, n, s, st);
  return launch_shapes<PairWide, PairDeep>(prm, d_maps, role, d_args, d_coefs, d_tiles, n, ends[1], s, st);
}

}  // namespace sf
