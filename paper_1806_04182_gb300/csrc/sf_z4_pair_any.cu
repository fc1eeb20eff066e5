// The two-point CCZ4 tile (sf_z4_pair.cuh) for patches of any size on the
// one-float row offset layout: runtime strides, tiles that overhang the patch
// with masked stores, one patch per launch (sf_z4_pair_batch.cu: the tiles of
// many patches).
//
// Three tile shapes of 512 points, 32 x 16 x 1, 32 x 8 x 2 and 16 x 8 x 4
// (kPairShapes).  Lanes outside the patch idle: with 32 x 16 x 1 tiles alone,
// 36% of them on patches of 16 to 64 points a side and 25% on 48^3 (96 mixed
// patches 11.6 ms per RK4 step, eight 48^3 patches with halo exchange 1.59; with
// the other two alone 10.0 and 1.36).  A launch takes rounds of one tile per
// SM, a round of the three shapes 40 : 41 : 43, and a last round that does not
// fill the SMs 0.7 to 0.95 of a full one, so a patch takes the shape of the
// least rounds x time.  Stage of 80 x 24 x 23 (138, 108 or 90 tiles: one
// round) 23.9, 24.0, 25.1 us; 48^3 (288, 288, 216) 47.5, 48.4, 51.7; 60 x 20 x 88
// (352, 264, 264) 69, 50, 55; 33 x 21 x 68 (272, 204, 153) 43, 42, 41; 70 x 50 x
// 61 (732, 651, 560) 113, 107, 96.  Over 60 sizes of 16 to 96 points a side the
// rule's shape takes 0.4% longer than the best of the three (the least tiles
// x time, 2.2%; 32 x 16 x 1 always, 8.6%) and none longer than 32 x 16 x 1.
#include <algorithm>

#include "sf_z4_pair.cuh"

namespace sf {

constexpr int kPairTime[3] = {40, 41, 43};  // of a round, relative
static long long pair_tiles(const sf_patch& p, int w) {
  long long n = 1;
  for (int d = 0; d < 3; ++d) n *= (p.n[d] + kPairShapes[w][d] - 1) / kPairShapes[w][d];
  return n;
}
static double pair_rounds(long long tiles) {
  const long long sms = std::max(1, sm_count()), full = tiles / sms, rest = tiles % sms;
  if (full == 0) return 1.0;
  return (double)full + (rest ? 0.7 + 0.25 * (double)rest / (double)sms : 0.0);
}

int z4_pair_shape(const sf_patch& p) {
  int best = 0;
  double cost = 0.0;
  for (int w = 0; w < 3; ++w) {
    const double c = pair_rounds(pair_tiles(p, w)) * kPairTime[w];
    if (w == 0 || c < cost) {
      cost = c;
      best = w;
    }
  }
  return best;
}

// The tiles of all patches of a launch share its rounds: one shape for all, or
// the wide or the deep one for each patch by its tiles x time.
void z4_pair_batch_shapes(const std::vector<const sf_patch*>& ps, std::vector<int>& shapes) {
  shapes.assign(ps.size(), 0);
  if (ps.empty()) return;
  double cost = 0.0;
  int best = 0;
  for (int w = 0; w < 3; ++w) {
    long long n = 0;
    for (const sf_patch* p : ps) n += pair_tiles(*p, w);
    const double c = pair_rounds(n) * kPairTime[w];
    if (w == 0 || c < cost) {
      cost = c;
      best = w;
    }
  }
  std::vector<int> mixed(ps.size());
  long long n = 0, work = 0;
  for (size_t q = 0; q < ps.size(); ++q) {
    const long long t1 = pair_tiles(*ps[q], 1), t2 = pair_tiles(*ps[q], 2);
    mixed[q] = t2 * kPairTime[2] < t1 * kPairTime[1] ? 2 : 1;
    n += mixed[q] == 2 ? t2 : t1;
    work += std::min(t2 * kPairTime[2], t1 * kPairTime[1]);
  }
  if (pair_rounds(n) * (double)work / (double)n < cost)
    shapes = mixed;
  else
    shapes.assign(ps.size(), best);
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
  switch (z4_pair_shape(p)) {
    case 0: return launch_any<PairFlat>(prm, p, s, stage, st);
    case 1: return launch_any<PairWide>(prm, p, s, stage, st);
    default: return launch_any<PairDeep>(prm, p, s, stage, st);
  }
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

}  // namespace sf
