// af_cube.cuh -- the arithmetic of scan-centric integration (Sec. 3.2), shared by
// the hashed map and the caller's dense box: one (return, cube voxel) pair from
// per-axis terms computed once per return.
//
// Every floating-point operation that decides an integer is an explicitly
// rounded IEEE single-precision operation, in the order the method states it;
// where a cheaper approximate value is used, it only takes decisions that the
// exact value is certain to agree with (margins of 2^-16).
#pragma once

#include "af_internal.cuh"

namespace af {

// Relative margin of decisions taken from approximate values: the reciprocal
// square root and two products are within 2^-20 for the normal arguments they
// are used on.
constexpr float kMargin = 1.52587890625e-05f;  // 2^-16

// The exact cone decision, RN(dot / RN(RN(sqrt(aa)) range)) > cone, out of
// line: it runs only within 2^-16 of the threshold, so divergent lanes call it
// instead of every lane carrying its instructions.
static __device__ __noinline__ bool cone_excludes_exact(float dot, float aa, float range, float cone) {
  return __fdiv_rn(dot, __fmul_rn(__fsqrt_rn(aa), range)) > cone;
}

template <int W>
struct CubeShape {
  static constexpr int C = W * W * W;                                 // offsets
  static constexpr int NT = ((C + 31) / 32) * 32 <= 1024 ? ((C + 31) / 32) * 32 : 1024;
  static constexpr int OPT = (C + NT - 1) / NT;                       // offsets per thread
  static constexpr int BA = (W + 6) / 8 + 1;                          // bricks per edge
  static constexpr int NB = BA * BA * BA;
  static constexpr int MR = W / 2;
};

// Returns per CTA ("tile") of one scan's integration: 4, 8, 12 or 16, the one that
// should take least time. An SM holds as many CTAs at once as their threads and
// registers allow (five of the cube of 7, one of 17) and takes the rest in turn; a
// CTA costs its pairs (offsets per thread times returns) and a setup (tables, per-axis
// terms) worth about six returns of one offset in the map's kernel, eight in the
// box's two. So small scans take the tile that spreads them over the chip in one go,
// large ones the tile that pays the setup least often without a last round for a few.
// Cubes of 3 and 5 have one and four warps per CTA, which a tile's setup keeps busy
// longer than its pairs: they stay with 4 and 8.
// Map's kernel, tiles of 4 / 8 / 12 / 16 (us): cube of 3, 6,000 returns 10.3 / 12.3 /
// 14.4 / 16.6; of 7, 6,000 returns 16.4 / 14.3 / 15.3 / 15.6, 12,000 25.0 / 21.1 /
// 22.0 / 20.2, 20,000 36.5 / 30.5 / 28.8 / 28.5, 60,000 90 / 72 / 67 / 63; of 9, 2,000
// returns 16.1 / 13.0 / 14.5 / 13.8, 4,000 24.4 / 19.6 / 20.1 / 17.4; of 17, 2,000
// returns 43 / 37 / 49 / 35, 20,000 308 / 270 / 248 / 260.
constexpr int kSetupMap = 6, kSetupBox = 8;
constexpr uint32_t kChipSMs = 152;

template <int W>
inline int tile_of(uint32_t n, int setup) {
  using S = CubeShape<W>;
  constexpr int most = W == 3 ? 4 : (W == 5 ? 8 : 16);
  constexpr uint32_t held = S::OPT > 3 ? 1 : (2048 / S::NT < 32 ? 2048 / S::NT : 32);
  int best = 0;
  uint64_t least = ~0ull;
  for (const int T : {8, 4, 12, 16}) {  // a tie keeps the one before
    if (T > most) continue;
    const uint32_t ctas = (n + T - 1) / T, turns = (ctas + kChipSMs - 1) / kChipSMs;
    const uint64_t cost = (uint64_t)(turns > held ? turns : held) * (uint64_t)(T * S::OPT + setup);
    if (cost < least) {
      least = cost;
      best = T;
    }
  }
  return best;
}

// What a pair reads of its return: x = range |p - q|, y = RN(1 / range) (for the
// approximate cone test), w = valid flag.
__device__ inline float4 return_record(float4 p, float q0, float q1, float q2) {
  float range = 0.f, ir = 0.f;
  if (p.w != 0.f) {
    const float b[3] = {__fsub_rn(p.x, q0), __fsub_rn(p.y, q1), __fsub_rn(p.z, q2)};
    range = __fsqrt_rn(
        __fadd_rn(__fadd_rn(__fmul_rn(b[0], b[0]), __fmul_rn(b[1], b[1])), __fmul_rn(b[2], b[2])));
    ir = __frcp_rn(range);
  }
  return make_float4(range, ir, 0.f, p.w);
}

// The rounded terms of one axis of the three sums a pair needs, (x - p)^2,
// (x - p)(p - q), (x - q)^2, for the voxel of absolute index i on that axis.
__device__ inline float4 axis_terms(const MapView& M, float pa, float qa, int i) {
  const float x = voxel_centre(i, M.v);
  const float a = __fsub_rn(x, pa), b = __fsub_rn(pa, qa), c = __fsub_rn(x, qa);
  return make_float4(__fmul_rn(a, a), __fmul_rn(a, b), __fmul_rn(c, c), 0.f);
}

// The contribution of a pair from its three axis records and its return's
// record, quantised; false if the cone excludes it. A pair adds three terms per
// sum in the order written (x, y, z), so every rounding is the same as computing
// it whole.
__device__ __forceinline__ bool pair_contribution(const MapView& M, const float4& tx, const float4& ty,
                                                  const float4& tz, const float4& pr, long long* dq) {
  const float tau = M.tau, cone = M.cone_cos;
  const float range = pr.x, ir = pr.y;
  const float aa = __fadd_rn(__fadd_rn(tx.x, ty.x), tz.x);
  // behind-surface cone: theta between x - p and p - q; excluded iff
  // RN(dot / RN(RN(sqrt(aa)) * range)) > cone
  if (aa > 0.f) {
    const float dot = __fadd_rn(__fadd_rn(tx.y, ty.y), tz.y);
    // dot <= 0 makes the rounded cosine <= 0, so with cone >= 0 it is kept
    if (dot > 0.f || cone < 0.f) {
      bool decided = false;
      if (aa > 1e-20f) {
        // a few ulp from the exact cosine (rsqrtf, two products, RN(1 / range))
        const float ca = dot * rsqrtf(aa) * ir;
        if (ca > cone + kMargin) return false;  // certainly excluded
        decided = ca < cone - kMargin;      // certainly kept
      }
      if (!decided && cone_excludes_exact(dot, aa, range, cone)) return false;
    }
  }
  // d = |p - q| - |x - q|, clamped to [0, tau] ([-tau, tau] in the ablation). The
  // exact root for every pair: a warp's voxels lie on both sides of the surface
  // and beyond tau, so screens that spared some lanes the root (|x - q| >= |p - q|,
  // or an approximate root beyond tau) cost every warp their branches as well
  // (31.9 against 26.7 us per pine frame, 84.8 against 68.0 us for 60,000 returns).
  const float cc = __fadd_rn(__fadd_rn(tx.z, ty.z), tz.z);
  const float d = fminf(fmaxf(__fsub_rn(range, __fsqrt_rn(cc)), M.dlo), tau);
  // |d| <= tau <= 1 m, so |d 2^20| < 2^31: the 32-bit conversion rounds
  // exactly as a 64-bit one would, and stays off the FP64 pipe
  *dq = (long long)__float2int_rn(__fmul_rn(d, kScale));
  return true;
}

}  // namespace af
