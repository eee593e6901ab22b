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

// Returns per CTA ("tile") of one scan's integration, by the scan's size. A tile's
// setup (brick table or box offsets, per-axis terms) is spread over its pairs, so
// larger tiles cost less a return as long as enough CTAs are left to overlap: with
// tiles of 8 / 12 / 16 the map's kernel takes 26.9 / 25.5 / 26.7 us for 20,000
// returns and 68.5 / 63.9 / 60.8 us for 60,000, the box's 27.6 / 27.0 / 26.3 us for
// 20,000. Small scans take small tiles, so that every SM has one.
constexpr int kTileSmall = 4, kTile = 12, kTileLarge = 16;
constexpr uint32_t kTileSmallBelow = 4000, kTileLargeFrom = 40000;

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
