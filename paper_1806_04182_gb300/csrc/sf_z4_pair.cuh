// CCZ4 stage kernel with two points per thread (Sec. V right-hand side with
// the Sec. II.B.1 stencils, fused with the RK stage of Sec. II.C), float
// storage, centred advection.
//
// Each thread computes two x-neighbours (i, i + 1), i even, and carries
// every quantity of the right-hand side as a pair (F2): each add, multiply
// and fused multiply-add of the per-point algebra is one .f32x2 instruction
// for both points, and so are most of the stencil operations.  The kernel
// is bound by instruction issue, so this halves the issue slots of the
// arithmetic, of the address and control work and of the ring waits per
// point.  It needs rows laid out so that points with even interior x sit on
// 8-byte boundaries: a row pitch of a multiple of 4 floats with one float
// before the first ghost point (arrays start 4 bytes past a 16-byte
// boundary).  Then every stencil read is a 64-bit shared-memory load of an
// aligned pair, and every RK read and write a 64-bit global access.
//
// Staging as in the one-point TMA kernel: a CTA of 8 warps computes a tile
// of 512 points (PairShape: 32 x 16 x 1, 32 x 8 x 2 or 16 x 8 x 4); the tile's
// box with a halo of 3 (4 along x) of every field is brought into a ring of
// shared memory slots by a cp.async.bulk.tensor load, fields in the order the
// right-hand side opens them, with a "full" mbarrier (TMA transaction count)
// and an "empty" mbarrier (one arrival per warp) per slot.  Every wait is
// bounded (about a second of clock cycles); a wait that gives up sets
// ST_TIMEOUT in the status word, the kernel finishes with whatever the slot
// holds, waits (bounded) for its own loads in flight and returns.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "sf_internal.cuh"
#include "sf_mbar.cuh"
#include "sf_z4.cuh"

namespace sf {

constexpr int kSY = 104, kSZ = 104 * 102;             // strides of the padded 96^3 layout
constexpr unsigned kPairWaitCycles = 2000000000u;   // ~1 s at GB300 clocks
constexpr int kPairWarps = 8;

// A tile of BX x BY x BZ = 512 points, two per thread, a ring of KS slots and
// RK inputs staged CHUNK fields at a time (three chunks hold the 25 fields).
// Threads take the tile's rows in order (rows of a plane, then the next
// plane), BX / 2 threads a row.  A 64-bit shared-memory read is served per
// half-warp: with rows of 40 floats its 16 threads read one row, with rows of
// 24 floats two rows, which must lie two apart (48 floats = 16 banks) to miss
// each other's banks.
template <int BX_, int BY_, int BZ_, int KS_, int CHUNK_>
struct PairShape {
  static constexpr int BX = BX_, BY = BY_, BZ = BZ_, KS = KS_, W = kPairWarps, kChunk = CHUNK_;
  static constexpr int XB = BX + 8, TY = BY + 6, TZ = BZ + 6;  // box, floats
  static constexpr int kBoxBytes = XB * TY * TZ * 4;
  static constexpr int kRkBoxBytes = 512 * kChunk * 4;
  static constexpr int kSlotBytes =
      ((kBoxBytes > kRkBoxBytes ? kBoxBytes : kRkBoxBytes) + 127) / 128 * 128;
  static constexpr int kSlotFloats = kSlotBytes / 4;
  static constexpr int kThreads = 32 * W;
  static constexpr int kBarOffset = KS * kSlotBytes;
  static constexpr int kRbufOffset = kBarOffset + 2 * KS * 8 + 16;  // (the give-up flag behind the barriers)
  static constexpr int kSmemBytes = kRbufOffset + 25 * kThreads * 8;
  static_assert(BX * BY * BZ == 2 * kThreads && (BX == 32 || (BX == 16 && BY % 4 == 0)), "tile");
  static_assert(kSmemBytes <= 232448 - 1024, "shared memory per CTA");
  static_assert(3 * kChunk >= 25, "three chunks cover the fields");
  // x offset and tile row of lane l of warp w, and the thread that owns (row, x)
  static __device__ __forceinline__ int lane_x(int l) { return 2 * (l % (BX / 2)); }
  static __device__ __forceinline__ int lane_row(int w, int l) {
    if constexpr (BX == 32) return 2 * w + (l >> 4);
    const int q = l >> 3;  // quarters take rows 0, 2, 1, 3
    return 4 * w + ((q & 1) * 2 + (q >> 1));
  }
  static __device__ __forceinline__ int owner(int row, int x) {
    if constexpr (BX == 32) return (row >> 1) * 32 + (row & 1) * 16 + (x >> 1);
    const int r = row & 3;
    return (row >> 2) * 32 + ((r & 1) * 2 + (r >> 1)) * 8 + (x >> 1);
  }
};

// 32 x 16 x 1, 7 slots: the compile-time layout.  Measured on the 96^3 patch
// against 6 warps with 9 slots (32 x 12 tiles; 2.35e9 against 2.81e9
// cell-updates/s), 5 slots (2.75e9), a persistent form in which one CTA per SM
// walks the tiles with the ring running on from tile to tile (1.84e9), and
// 32 x 8 x 2 with 7 to 9 slots (1130 against 990 us per step: twice the
// instruction-cache misses).
//
// An SM streams instructions at full rate from 128 KB (measured: straight code
// of 128 KB 1.5 cycles per instruction with two warps a scheduler, of 136 KB
// 2.4, of 160 KB 3.2), so the ring's waits and loads are written to stay small:
// compact waits with uniform branches, loads issued by an elected lane, and
// field pointers stepped in the write phase took the kernel from 135 to 122 KB
// and from 7310 to 6960 warp instructions per warp (96^3 step 985 -> 970 us,
// sub-cycled 64^3 pair 1667 -> 1555 us).
using PairFlat = PairShape<32, 16, 1, 7, 12>;
// 8 slots for the tiles of several planes (9, 7 and 5: 3%, 1% and 4% slower on eight 48^3 patches)
using PairWide = PairShape<32, 8, 2, 8, 9>;
using PairDeep = PairShape<16, 8, 4, 8, 9>;

// Order in which z4_rhs opens the fields' stencils.  Without the
// Gamma-driver (shift frozen) the last three are not used.
static __constant__ signed char kPairFieldSeq[25] = {19, 20, 21, 1, 2, 3, 4, 5, 6, 14, 15, 16, 0,
                                                     18, 7, 17, 8, 9, 10, 11, 12, 13, 22, 23, 24};

// Stencil weights as broadcast pairs (Sec. II.B.1), per direction d.
struct PairCoef {
  F2 d1[3], d2[3];         // D_d = (U+1 - U-1) d1 + (U-2 - U+2) d2: 8/(12 h), 1/(12 h)
  F2 k1[3], k2[3], k3[3];  // KO: 15 s, -6 s, s on the sums at distance 1, 2, 3
  F2 kc;                   // KO centre: -20 (s_x + s_y + s_z), s = sigma / (64 h)
  F2 e1[3], e2[3], e0[3];  // D_dd: 16 e, -e, -30 e with e = 1 / (12 h^2)
  F2 mx[3][3];             // mixed (xy, xz, yz): w, 8 w, 64 w with w = 1 / (144 h_a h_b)
};

inline PairCoef pair_coef(const sf_params& prm, const sf_patch& p) {
  PairCoef c;
  double kc = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double h = p.dx[d], s = prm.sigma_ko / (64.0 * h), e = 1.0 / (12.0 * h * h);
    auto b = [](double v) { F2 r; r.x = r.y = float(v); return r; };
    c.d1[d] = b(8.0 / (12.0 * h));
    c.d2[d] = b(1.0 / (12.0 * h));
    c.k1[d] = b(15.0 * s);
    c.k2[d] = b(-6.0 * s);
    c.k3[d] = b(s);
    kc += s;
    c.e1[d] = b(16.0 * e);
    c.e2[d] = b(-e);
    c.e0[d] = b(-30.0 * e);
  }
  c.kc.x = c.kc.y = float(-20.0 * kc);
  const double w[3] = {1.0 / (144.0 * p.dx[0] * p.dx[1]), 1.0 / (144.0 * p.dx[0] * p.dx[2]),
                       1.0 / (144.0 * p.dx[1] * p.dx[2])};
  for (int m = 0; m < 3; ++m)
    for (int k = 0; k < 3; ++k) c.mx[m][k].x = c.mx[m][k].y = float(w[m] * (k == 0 ? 1.0 : k == 1 ? 8.0 : 64.0));
  return c;
}

__device__ __forceinline__ void tma_load_4d(float* dst, const CUtensorMap* map, int x, int y, int z,
                                            int f, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(saddr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(f), "r"(saddr(bar))
      : "memory");
}

// Stencil source of z4_rhs for the pair of points (i, i + 1): the staged
// boxes in shared memory, the centre values (all fields, at the start) from
// global memory.
template <typename C, int NARR = 0>
struct PairSrc {
  static constexpr int KS = C::KS;
  static constexpr int kY = C::XB;            // box row, floats
  static constexpr int kZ = C::XB * C::TY;    // box plane, floats
  const float* u;  // global stage input at point i, field 0
  long long F;
  const PairCoef* pc;
  float* tiles;
  uint64_t* full;
  uint64_t* empty;
  unsigned* gaveup;  // shared flag: some wait of the CTA gave up
  const CUtensorMap* map;
  unsigned* status;
  int local;  // this thread's point i inside a box (an even float index)
  int use, cur, nuses, issued, next;
  int gx, gy, gz;  // tensor coordinates of the box origin
  int warp;        // warp index, uniform
  // NARR > 0: after the nfu field uses, the RK inputs of the tile (NARR
  // arrays) follow as uses of the ring, 3 chunks of kChunk fields per array,
  // chunk-major, from the maps rkmap[0 .. NARR - 1] at tensor coordinates
  // (rx, ry, rz); consumed by the write phase (acquire / release)
  int nfu;
  const CUtensorMap* rkmap;
  int rx, ry, rz;

  // warp 0: load use j into its slot once the previous occupant (use j - KS)
  // has been released by every warp.  The whole warp waits and one elected lane
  // issues: in a region that a lane-index test opens, the wait and the issue
  // compile to loops over the active lanes (1 KB of code per site).  FIELD: use
  // j is a field whatever nfu is.
  template <bool FIELD>
  __device__ __forceinline__ void issue(int j) {
    const int sl = j % KS;
    if (!FIELD && j >= nuses) return;
    if (j >= KS) mbar_wait_warp(&empty[sl], ((j / KS) - 1) & 1, kPairWaitCycles, gaveup);
    if (elect_one() && !*reinterpret_cast<volatile unsigned*>(gaveup)) {
      const CUtensorMap* m = map;
      int x = gx, y = gy, z = gz, f = kPairFieldSeq[FIELD ? j : min(j, 24)];
      unsigned bytes = C::kBoxBytes;
      if constexpr (!FIELD && NARR > 0) {
        if (j >= nfu) {
          const int r = j - nfu;
          m = rkmap + r % NARR;
          x = rx; y = ry; z = rz; f = C::kChunk * (r / NARR);
          bytes = C::kRkBoxBytes;
        }
      }
      mbar_expect(&full[sl], bytes);
      tma_load_4d(tiles + sl * C::kSlotFloats, m, x, y, z, f, &full[sl]);
      issued = j + 1;
    }
    __syncwarp();
  }
  // write phase: wait for RK use i (kept until release(i)), after issuing
  // the uses up to i + KS - NARR (their slots' previous uses are released)
  __device__ __forceinline__ const float* acquire(int i) {
    if (warp == 0) {
#pragma unroll 1
      for (; next <= i + KS - NARR && next < nuses; ++next) issue<false>(next);
    }
    mbar_wait_warp(&full[i % KS], (i / KS) & 1, kPairWaitCycles, gaveup);
    return tiles + (i % KS) * C::kSlotFloats;
  }
  __device__ __forceinline__ void release(int i) {
    __syncwarp();
    mbar_arrive_warp(&empty[i % KS]);
  }
  __device__ __forceinline__ void prologue() {
    if (warp == 0) {
#pragma unroll 1
      for (int j = 0; j < KS - 1; ++j) issue<true>(j);
    }
  }
  __device__ __forceinline__ void begin() {
    const int i = use++;
    if (i > 0) {
      if (warp == 0) {
        if (i + KS - 2 < 22)
          issue<true>(i + KS - 2);
        else
          issue<false>(i + KS - 2);
      }
      release(i - 1);
    }
    cur = i % KS;
    mbar_wait_warp(&full[cur], (i / KS) & 1, kPairWaitCycles, gaveup);
  }
  // end of the field uses (z4_rhs's last call): with staged RK inputs the
  // last field's slot is released for them
  __device__ __forceinline__ void finish() {
    next = use + KS - 2;  // (uses up to use + KS - 3 have been issued)
    if constexpr (NARR > 0)
      release(use - 1);
    else
      final_finish();
  }
  // if a wait gave up: report it, and the leader waits (bounded) for the last
  // load of every slot, so that none is in flight when the CTA exits
  __device__ __forceinline__ void final_finish() {
    if (*reinterpret_cast<volatile unsigned*>(gaveup)) {
      atomicOr(status, ST_TIMEOUT);
      // (in the one lane that issued; in the others `issued` is 0)
      for (int j = max(0, issued - KS); j < issued; ++j)
        mbar_wait(&full[j % KS], (j / KS) & 1, kPairWaitCycles);
    }
  }

  __device__ __forceinline__ const float* box() const { return tiles + cur * C::kSlotFloats + local; }
  // aligned pair at float offset o (even) from point i
  static __device__ __forceinline__ F2 L(const float* p, int o) { return *reinterpret_cast<const F2*>(p + o); }

  __device__ __forceinline__ F2 centre(int f) const {
    return *reinterpret_cast<const F2*>(u + f * F);
  }

  // 19-point cross of both points.  Along x the neighbours at odd distance
  // straddle two aligned pairs: their sums and differences are formed lane
  // by lane (two scalar instructions straight into a pair), everything else
  // on pairs.
  __device__ __forceinline__ Cross<F2> cross(int f, bool second) {
    begin();
    const float* p = box();
    const PairCoef& c = *pc;
    const F2 am4 = L(p, -4), am2 = L(p, -2), a0 = L(p, 0), a2 = L(p, 2), a4 = L(p, 4);
    // x: values q(o) at offset o from point i; point i + 1 reads q(o + 1)
    const F2 xs1(am2.y + a0.y, a0.x + a2.x);   // U-1 + U+1
    const F2 xd1(a0.y - am2.y, a2.x - a0.x);   // U+1 - U-1
    const F2 xs3(am4.y + a2.y, am2.x + a4.x);  // U-3 + U+3
    const F2 xs2 = add2(am2, a2), xd2 = sub2(am2, a2);
    const F2 ym1 = L(p, -kY), yp1 = L(p, kY), ym2 = L(p, -2 * kY), yp2 = L(p, 2 * kY),
             ym3 = L(p, -3 * kY), yp3 = L(p, 3 * kY);
    const F2 zm1 = L(p, -kZ), zp1 = L(p, kZ), zm2 = L(p, -2 * kZ), zp2 = L(p, 2 * kZ),
             zm3 = L(p, -3 * kZ), zp3 = L(p, 3 * kZ);
    const F2 ys1 = add2(ym1, yp1), yd1 = sub2(yp1, ym1), ys2 = add2(ym2, yp2), yd2 = sub2(ym2, yp2),
             ys3 = add2(ym3, yp3);
    const F2 zs1 = add2(zm1, zp1), zd1 = sub2(zp1, zm1), zs2 = add2(zm2, zp2), zd2 = sub2(zm2, zp2),
             zs3 = add2(zm3, zp3);
    Cross<F2> x;
    x.c = a0;
    x.d[0] = fma2(xd1, c.d1[0], mul2(xd2, c.d2[0]));
    x.d[1] = fma2(yd1, c.d1[1], mul2(yd2, c.d2[1]));
    x.d[2] = fma2(zd1, c.d1[2], mul2(zd2, c.d2[2]));
    F2 ko = mul2(a0, c.kc);
    ko = fma2(xs3, c.k3[0], ko);
    ko = fma2(ys3, c.k3[1], ko);
    ko = fma2(zs3, c.k3[2], ko);
    ko = fma2(xs2, c.k2[0], ko);
    ko = fma2(ys2, c.k2[1], ko);
    ko = fma2(zs2, c.k2[2], ko);
    ko = fma2(xs1, c.k1[0], ko);
    ko = fma2(ys1, c.k1[1], ko);
    x.ko = fma2(zs1, c.k1[2], ko);
    if (second) {
      x.dd[0] = fma2(xs1, c.e1[0], fma2(xs2, c.e2[0], mul2(a0, c.e0[0])));
      x.dd[1] = fma2(ys1, c.e1[1], fma2(ys2, c.e2[1], mul2(a0, c.e0[1])));
      x.dd[2] = fma2(zs1, c.e1[2], fma2(zs2, c.e2[2], mul2(a0, c.e0[2])));
    } else {
      x.dd[0] = x.dd[1] = x.dd[2] = F2(0.0f);
    }
    x.adv = F2(0.0f);
    return x;
  }

  // D_xb with b = y (s = kY) or z (s = kZ): with r1(o) = U(-2) - U(+2) and
  // r8(o) = U(+1) - U(-1) along x in the row at offset o across,
  // D_xb = w (r1(-2) - r1(2)) + 8 w (r8(-2) - r8(2) + r1(1) - r1(-1)) + 64 w (r8(1) - r8(-1)).
  __device__ __forceinline__ F2 mix_x(const float* p, int s, const F2* w) const {
    F2 r1[4], r8[4];  // rows -2, -1, 1, 2
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = (q < 2 ? q - 2 : q - 1) * s;
      const F2 am2 = L(p, o - 2), a0 = L(p, o), a2 = L(p, o + 2);
      r1[q] = sub2(am2, a2);
      r8[q] = F2(a0.y - am2.y, a2.x - a0.x);
    }
    const F2 x1 = sub2(r1[0], r1[3]);
    const F2 x8 = add2(sub2(r8[0], r8[3]), sub2(r1[2], r1[1]));
    const F2 x64 = sub2(r8[2], r8[1]);
    return fma2(x64, w[2], fma2(x8, w[1], mul2(x1, w[0])));
  }
  // D_yz: the same along y, rows across in z
  __device__ __forceinline__ F2 mix_yz(const float* p, const F2* w) const {
    F2 r1[4], r8[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int o = (q < 2 ? q - 2 : q - 1) * kZ;
      r1[q] = sub2(L(p, o - 2 * kY), L(p, o + 2 * kY));
      r8[q] = sub2(L(p, o + kY), L(p, o - kY));
    }
    const F2 x1 = sub2(r1[0], r1[3]);
    const F2 x8 = add2(sub2(r8[0], r8[3]), sub2(r1[2], r1[1]));
    const F2 x64 = sub2(r8[2], r8[1]);
    return fma2(x64, w[2], fma2(x8, w[1], mul2(x1, w[0])));
  }
  // mixed derivatives (xy, xz, yz) of the field whose cross was just read
  __device__ __forceinline__ void mix3(int, F2* out) const {
    const float* p = box();
    out[0] = mix_x(p, kY, pc->mx[0]);
    out[1] = mix_x(p, kZ, pc->mx[1]);
    out[2] = mix_yz(p, pc->mx[2]);
  }
};

// Forms of the RK combination fixed at compile time: the kernel is
// instantiated per form, so that its write phase carries one form's code and
// no branches on the stage (the generic form decides at run time).
//   kRk4First: RK4 stage 0 with the Kahan accumulator (U^n = the stage input)
//   kRk4Mid:   RK4 stages 1 and 2
//   kRk4Last:  RK4 stage 3 with the Kahan compensation
enum : int { kRkGeneric = 0, kRk4First = 1, kRk4Mid = 2, kRk4Last = 3 };

inline int rk_form(const StageArgs& s) {
  if (s.mode != 0 || s.rk != SF_RK4 || !s.kahan) return kRkGeneric;
  if (s.stage == 0) return s.un_alias ? kRk4First : kRkGeneric;
  return s.stage < 3 ? kRk4Mid : kRk4Last;
}

// Store of a value pair; MASKED (tiles that overhang the patch): vm bit 0
// for point i, bit 1 for point i + 1 (never set without bit 0).
template <bool MASKED>
__device__ __forceinline__ void store2(float* p, F2 v, unsigned vm) {
  if constexpr (MASKED) {
    if (vm == 3u) *reinterpret_cast<F2*>(p) = v;
    else if (vm & 1u) p[0] = v.x;
  } else {
    *reinterpret_cast<F2*>(p) = v;
  }
}

// RK stage combination of one field value pair (sf_common.cuh's
// stage_combine on pairs), the stage known at run time: writes the
// accumulator / Kahan term and returns the next stage input.
__device__ __forceinline__ F2 stage_combine2(const PatchArgs<float>& a, const StageArgs& s,
                                             long long o, F2 centre, F2 un_m, F2 acc, F2 kh, F2 r) {
  const F2 cn(a.c_next), ca(a.c_acc);
  const F2 un = s.un_alias ? centre : un_m;
  F2 out;
  if (s.rk == SF_RK4) {
    if (s.stage == 0) {
      *reinterpret_cast<F2*>(a.acc + o) = s.kahan ? mul2(ca, r) : fma2(ca, r, un);
      out = fma2(cn, r, un);
    } else if (s.stage < 3) {
      *reinterpret_cast<F2*>(a.acc + o) = fma2(ca, r, acc);
      out = fma2(cn, r, un);
    } else if (!s.kahan) {
      out = fma2(cn, r, acc);
    } else {
      const F2 inc = fma2(cn, r, acc);
      const F2 y = sub2(inc, kh);
      const F2 t = add2(un, y);
      *reinterpret_cast<F2*>(a.kh + o) = sub2(sub2(t, un), y);
      out = t;
    }
  } else {
    const F2 dt(a.dt);
    if (s.stage == 0) out = fma2(dt, r, un);
    else if (s.stage == 1) out = fma2(F2(0.75f), un, mul2(F2(0.25f), fma2(dt, r, centre)));
    else out = fma2(un, F2(float(1.0 / 3.0)), mul2(F2(float(2.0 / 3.0)), fma2(dt, r, centre)));
  }
  return out;
}

// The stage write of the 25 fields of both points, right-hand sides parked
// in shared memory (r[f * stride]); the scheme of write_fields (batches of
// five fields with every read issued before the writes, periodic images of
// boundary points in one rolled pass at the end) on 64-bit accesses.
__device__ __forceinline__ void write_fields_pair(const PatchArgs<float>& a, const StageArgs& s,
                                                  long long c, int i, int j, int k, F2* r,
                                                  int stride) {
  if (s.mode == 1) {
    const long long oi = ((long long)k * a.n[1] + j) * a.n[0] + i;
#pragma unroll 1
    for (int f = 0; f < 25; ++f) {
      const F2 v = r[f * stride];
      a.nx[f * a.ninterior + oi] = v.x;
      a.nx[f * a.ninterior + oi + 1] = v.y;
    }
    return;
  }
  const bool rk4 = s.rk == SF_RK4;
  const bool need_centre = s.un_alias || !rk4, need_un = !s.un_alias;
  const bool need_acc = rk4 && s.stage > 0, need_kh = rk4 && s.stage == 3 && s.kahan;
  auto ld = [](const float* q) { return *reinterpret_cast<const F2*>(q); };
#pragma unroll 1
  for (int f0 = 0; f0 < 25; f0 += 5) {
    F2 cen[5], un[5], acc[5], kh[5], rr[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const long long o = (f0 + q) * a.sf + c;
      rr[q] = r[(f0 + q) * stride];
      cen[q] = need_centre ? ld(a.us + o) : F2(0.0f);
      un[q] = need_un ? ld(a.un + o) : F2(0.0f);
      acc[q] = need_acc ? ld(a.acc + o) : F2(0.0f);
      kh[q] = need_kh ? ld(a.kh + o) : F2(0.0f);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const long long o = (f0 + q) * a.sf + c;
      const F2 out = stage_combine2(a, s, o, cen[q], un[q], acc[q], kh[q], rr[q]);
      *reinterpret_cast<F2*>(a.nx + o) = out;
      if (s.check_finite && !(finite_(out.x) && finite_(out.y))) atomicOr(s.status, ST_NONFINITE);
      r[(f0 + q) * stride] = out;
    }
  }
}

// The y and z periodic images of the pair's new values (rows and planes next
// to a face; r holds the values written), as aligned pairs: a shift in y or z
// keeps the pair on its 8-byte boundary.  The x ghost columns are written by
// write_x_images (RK4 forms) or by pair_xghost_kernel after the stage.
template <bool MASKED = false>
__device__ __forceinline__ void write_yz_images(const PatchArgs<float>& a, const StageArgs& s,
                                                long long c, int i, int j, int k, const F2* r,
                                                int stride, unsigned vm = 3u) {
  if (MASKED && !(vm & 1u)) return;
  const unsigned m = ghost_images(a, s, i, j, k).mask & ~3u;
  if (!m) return;
#pragma unroll 1
  for (int f = 0; f < 25; ++f) {
    const F2 v = r[f * stride];
    float* q = a.nx + f * a.sf + c;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      if (p && !(m & (p == 1 ? 16u : 32u))) continue;
      const long long oz = p == 0 ? 0 : (p == 1 ? 1 : -1) * (long long)a.n[2] * a.sz;
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        if (w && !(m & (w == 1 ? 4u : 8u))) continue;
        const long long oy = w == 0 ? 0 : (w == 1 ? 1 : -1) * (long long)a.n[1] * a.sy;
        if (p | w) store2<MASKED>(q + oz + oy, v, vm);
      }
    }
  }
}

// The x periodic images of the patch's boundary columns that lie in a tile
// (lower corner x0, y0, z0), written by the CTA from the
// tile's new values in shared memory (r: the pair of thread t for field f at
// r[f * stride + t]).  Interior x = 0..2 go to ghost x = n0 .. n0 + 2 (past
// the interior), x = n0 - 3 .. n0 - 1 to x = -3 .. -1; each also at the y and
// z image rows of its point, so that with write_yz_images every ghost value
// of the tile's points is written.  Spread over the CTA's threads.
template <typename C>
__device__ __forceinline__ void write_x_images(const PatchArgs<float>& a, const StageArgs& s,
                                               int x0, int y0, int z0, const F2* r, int stride,
                                               int tid) {
  const int n0 = a.n[0];
  const int lo0 = x0, lo1 = min(min(3, n0), x0 + C::BX);          // columns with an image at +n0
  const int hi0 = max(n0 - 3, x0), hi1 = min(n0, x0 + C::BX);      // columns with an image at -n0
  const int nlo = max(0, lo1 - lo0), nhi = max(0, hi1 - hi0), ncol = nlo + nhi;
  if (!ncol) return;
  constexpr int R = C::BY * C::BZ;  // tile rows
#pragma unroll 1
  for (int v = tid; v < ncol * R * 25; v += stride) {
    const int f = v / (ncol * R), rem = v - f * (ncol * R), row = rem / ncol, cc = rem - row * ncol;
    const int j = y0 + row % C::BY, k = z0 + row / C::BY;
    if (j >= a.n[1] || (C::BZ > 1 && k >= a.n[2])) continue;
    const bool low = cc < nlo;
    const int x = low ? lo0 + cc : hi0 + (cc - nlo);
    const int xl = x - x0;  // tile-local x of the source point
    const F2 pr = r[f * stride + C::owner(row, xl)];
    const float val = (xl & 1) ? pr.y : pr.x;
    const unsigned m = ghost_images(a, s, x, j, k).mask;
    const long long o = f * a.sf + (long long)(k + 3) * a.sz + (long long)(j + 3) * a.sy + (x + 3) +
                        (low ? n0 : -n0);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      if (p && !(m & (p == 1 ? 16u : 32u))) continue;
      const long long oz = p == 0 ? 0 : (p == 1 ? 1 : -1) * (long long)a.n[2] * a.sz;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (q && !(m & (q == 1 ? 4u : 8u))) continue;
        const long long oy = q == 0 ? 0 : (q == 1 ? 1 : -1) * (long long)a.n[1] * a.sy;
        a.nx[o + oz + oy] = val;
      }
    }
  }
}

// The stage write with the RK inputs staged in the ring (the specialised
// forms): per block of kChunk fields, the chunks of the NARR input arrays
// are acquired, every field of the block combined and stored, and the
// chunks released.  Array order: kRk4First: u_stage (= U^n); kRk4Mid: U^n,
// accumulator; kRk4Last: U^n, accumulator, Kahan term.
template <typename C, int FORM, int NARR, bool MASKED = false, typename Src>
__device__ __forceinline__ void write_fields_staged(const PatchArgs<float>& a, const StageArgs& s,
                                                    long long c, F2* r, int stride, Src& src,
                                                    int lpos, unsigned vm = 3u) {
  static_assert(NARR >= 1 && NARR <= 3, "staged arrays");
  auto ld = [](const float* q) { return *reinterpret_cast<const F2*>(q); };
  bool bad = false;  // a non-finite value written (reported once, at the end)
  // element pointers that step by a field: the next stage input, and the array
  // the form updates (accumulator, or the Kahan term)
  float* nx = a.nx + c;
  float* aux = (FORM == kRk4Last ? a.kh : a.acc) + c;
  const F2 cn(a.c_next), ca(a.c_acc);
#pragma unroll 1
  for (int blk = 0; blk < 3; ++blk) {
    const float* in[NARR];
#pragma unroll
    for (int t = 0; t < NARR; ++t) in[t] = src.acquire(src.nfu + blk * NARR + t) + lpos;
    const int nf = min(C::kChunk, 25 - C::kChunk * blk);
#pragma unroll 1
    for (int q = 0; q < nf; ++q) {
      const F2 v0 = ld(in[0]);
      const F2 v1 = NARR > 1 ? ld(in[NARR > 1 ? 1 : 0]) : F2(0.0f);
      const F2 v2 = NARR > 2 ? ld(in[NARR > 2 ? 2 : 0]) : F2(0.0f);
      const F2 rr = *r;
      // stage_combine2 of the form (the first array is U^n)
      F2 out;
      if constexpr (FORM == kRk4First) {
        store2<MASKED>(aux, mul2(ca, rr), vm);
        out = fma2(cn, rr, v0);
      } else if constexpr (FORM == kRk4Mid) {
        store2<MASKED>(aux, fma2(ca, rr, v1), vm);
        out = fma2(cn, rr, v0);
      } else {
        const F2 y = sub2(fma2(cn, rr, v1), v2);
        out = add2(v0, y);
        store2<MASKED>(aux, sub2(sub2(out, v0), y), vm);
      }
      store2<MASKED>(nx, out, vm);
      if (s.check_finite) {
        if constexpr (MASKED)
          bad |= ((vm & 1u) && !finite_(out.x)) || ((vm & 2u) && !finite_(out.y));
        else
          bad |= !(finite_(out.x) && finite_(out.y));
      }
      *r = out;
      r += stride;
      nx += a.sf;
      aux += a.sf;
#pragma unroll
      for (int t = 0; t < NARR; ++t) in[t] += 512;
    }
#pragma unroll
    for (int t = 0; t < NARR; ++t) src.release(src.nfu + blk * NARR + t);
  }
  if (s.check_finite && bad) atomicOr(s.status, ST_NONFINITE);
}

// Tensor maps of the RK input arrays of a stage form (unused ones zero).
struct RkMaps {
  CUtensorMap m[3];
};

// One tile with lower corner (x0, y0, z0): the stencil
// boxes staged through the ring, the right-hand side, the stage write and the
// periodic images of its points.  BATCH: the patch's strides come from `a`
// and the tile may overhang the patch (points outside write nothing, their
// centre reads are clamped into the patch); otherwise the compile-time
// strides of the padded 96^3-class layout and whole tiles.
template <typename H2, typename C, int FORM, bool BATCH>
__device__ __forceinline__ void pair_tile(const CUtensorMap* map, const CUtensorMap* rkmaps,
                                          const PatchArgs<float>& a, const StageArgs& s,
                                          const Z4Coef<float>& zc, const PairCoef* pc, int x0,
                                          int y0, int z0, unsigned char* smem) {
  constexpr int NARR = FORM == kRk4First ? 1 : (FORM == kRk4Mid ? 2 : (FORM == kRk4Last ? 3 : 0));
  static_assert(!BATCH || NARR > 0, "batched tiles take the RK4 stage forms");
  constexpr int W = C::W, KS = C::KS;
  float* tiles = reinterpret_cast<float*>(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kBarOffset);
  uint64_t* empty = full + KS;
  unsigned* gaveup = reinterpret_cast<unsigned*>(empty + KS);
  const int tid = threadIdx.y * 32 + threadIdx.x;
  if (tid == 0) {
    for (int q = 0; q < KS; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], W);
    }
    *gaveup = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  wait_predecessor();
  __syncthreads();
  const int px = C::lane_x(threadIdx.x);
  const int lr = C::lane_row(threadIdx.y, threadIdx.x);  // row of the tile
  const int ly = C::BZ == 1 ? lr : lr % C::BY, lz = C::BZ == 1 ? 0 : lr / C::BY;
  const int i = x0 + px;
  const int j = y0 + ly;
  const int k = z0 + lz;
  long long c;
  unsigned vm = 3u;  // bit 0: point i in the patch, bit 1: point i + 1
  if constexpr (BATCH) {
    vm = j < a.n[1] && (C::BZ == 1 || k < a.n[2])
             ? (i < a.n[0] ? 1u : 0u) | (i + 1 < a.n[0] ? 2u : 0u)
             : 0u;
    const int ic = min(i, (a.n[0] - 1) & ~1), jc = min(j, a.n[1] - 1);
    const int kc = C::BZ == 1 ? k : min(k, a.n[2] - 1);
    c = (long long)(kc + 3) * a.sz + (long long)(jc + 3) * a.sy + (ic + 3);
  } else {
    c = (long long)(k + 3) * kSZ + (long long)(j + 3) * kSY + (i + 3);
  }
  if (NARR == 0 && C::BX == 32 && (threadIdx.x & 15) == 0 && s.mode == 0) {
    // generic form (RK inputs read from global memory in the write phase):
    // the row's 32 points start on a 16-byte boundary, prefetch their 128 B
    // of every field the RK combination reads.  The RK4 forms stage those
    // inputs through the TMA ring, where a prefetch only competes with the
    // stencil boxes.
    if (!s.un_alias) prefetch_rows<128>(a.un + c, a.sf);
    if (s.rk == SF_RK4 && s.stage > 0) prefetch_rows<128>(a.acc + c, a.sf);
    if (s.kahan && s.stage == 3) prefetch_rows<128>(a.kh + c, a.sf);
  }
  PairSrc<C, NARR> src;
  src.u = a.us + c;
  src.F = a.sf;
  src.pc = pc;
  src.tiles = tiles;
  src.full = full;
  src.empty = empty;
  src.gaveup = gaveup;
  src.map = map;
  src.status = s.status;
  src.local = ((lz + 3) * C::TY + ly + 3) * C::XB + px + 4;
  src.use = 0;
  src.cur = 0;
  src.nfu = zc.shift_frozen ? 22 : 25;
  src.nuses = src.nfu + 3 * NARR;
  src.rkmap = rkmaps;
  src.rx = x0 + 4;  // tensor x = ghosted x + 1 of point x0
  src.ry = y0 + 3;
  src.rz = z0 + 3;
  src.issued = 0;
  src.gx = x0;  // tensor x = ghosted x + 1; the box starts 4 before point x0
  src.gy = y0;
  src.gz = z0;
  src.warp = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0);
  src.prologue();
  F2* rbuf = reinterpret_cast<F2*>(smem + C::kRbufOffset);
  F2 be[3];
  z4_rhs<F2, H2, false>(zc, src, be, [&](int f, F2 r, F2) { rbuf[f * C::kThreads + tid] = r; });
  if constexpr (NARR > 0)
    write_fields_staged<C, FORM, NARR, BATCH>(a, s, c, rbuf + tid, C::kThreads, src, lr * C::BX + px, vm);
  else
    write_fields_pair(a, s, c, i, j, k, rbuf + tid, C::kThreads);
  write_yz_images<BATCH>(a, s, c, i, j, k, rbuf + tid, C::kThreads, vm);
  if constexpr (NARR > 0) {
    if (s.ghosts && s.mode == 0) {
      __syncthreads();  // every new value of the tile is in rbuf
      write_x_images<C>(a, s, x0, y0, z0, rbuf, C::kThreads, tid);
    }
    src.final_finish();
  }
}

inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn_pair() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

inline bool offset_aligned(const void* q) {
  return q && reinterpret_cast<uintptr_t>(q) % 16 == 4;
}

// Tensor maps over the arrays of a patch: tensor x = ghosted x + 1 (the map
// starts at the float before ghost point 0).  A stencil box of shape C, or its
// box of RK inputs.
template <typename C>
sf_status encode_pair_map(CUtensorMap* m, const sf_patch& p, const void* array, bool rk) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn_pair();
  if (!enc) return set_error(SF_ECUDA, "cuTensorMapEncodeTiled not available");
  memset(m, 0, sizeof(*m));
  const cuuint64_t dims[4] = {(cuuint64_t)(p.n[0] + 7), (cuuint64_t)(p.n[1] + 6),
                              (cuuint64_t)(p.n[2] + 6), 25};
  const cuuint64_t strides[3] = {(cuuint64_t)p.sy * 4, (cuuint64_t)p.sz * 4, (cuuint64_t)p.sf * 4};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const cuuint32_t sbox[4] = {C::XB, C::TY, C::TZ, 1};
  const cuuint32_t rbox[4] = {C::BX, C::BY, C::BZ, C::kChunk};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
                         static_cast<char*>(const_cast<void*>(array)) - 4, dims, strides,
                         rk ? rbox : sbox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(SF_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return SF_OK;
}

// The arrays that a stage form stages through the ring.
template <typename C>
sf_status encode_rk_maps(RkMaps* rk, const sf_patch& p, int form) {
  memset(rk, 0, sizeof(*rk));
  const void* arrs[3] = {nullptr, nullptr, nullptr};
  if (form == kRk4First) arrs[0] = p.u_stage;
  if (form == kRk4Mid || form == kRk4Last) {
    arrs[0] = p.u_n;
    arrs[1] = p.acc;
  }
  if (form == kRk4Last) arrs[2] = p.kahan;
  for (int q = 0; q < 3; ++q)
    if (arrs[q])
      if (sf_status e = encode_pair_map<C>(&rk->m[q], p, arrs[q], true)) return e;
  return SF_OK;
}

}  // namespace sf
