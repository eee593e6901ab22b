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

// Approximate square root (MUFU reciprocal square root), relative error well
// below 2^-20 for the normal arguments it is used on. Only ever used to take
// a decision that the exact result is certain to agree with (margins of
// 2^-16 relative); near any threshold the exact IEEE operation decides.
__device__ inline float sqrt_approx(float x) { return x * rsqrtf(x); }

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

// What a pair reads of its return: range |p - q|, RN(|p - q|^2), RN(1 / range)
// (for the approximate cone test), valid flag.
__device__ inline float4 return_record(float4 p, float q0, float q1, float q2) {
  float bb = 0.f, range = 0.f, ir = 0.f;
  if (p.w != 0.f) {
    const float b[3] = {__fsub_rn(p.x, q0), __fsub_rn(p.y, q1), __fsub_rn(p.z, q2)};
    bb = __fadd_rn(__fadd_rn(__fmul_rn(b[0], b[0]), __fmul_rn(b[1], b[1])), __fmul_rn(b[2], b[2]));
    range = __fsqrt_rn(bb);
    ir = __frcp_rn(range);
  }
  return make_float4(range, bb, ir, p.w);
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
  const float range = pr.x, bb = pr.y, ir = pr.z;
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
  // d = |p - q| - |x - q|, clamped to [0, tau] ([-tau, tau] in the ablation)
  const float cc = __fadd_rn(__fadd_rn(tx.z, ty.z), tz.z);
  float d;
  if (cc >= bb && !M.clamp_signed) {
    d = 0.f;  // |x - q| >= |p - q|: the rounded difference is <= 0
  } else if (cc > 1e-20f && range - sqrt_approx(cc) > tau + range * kMargin) {
    d = tau;  // the exact difference exceeds tau
  } else {
    d = __fsub_rn(range, __fsqrt_rn(cc));
    d = d < M.dlo ? M.dlo : d;
    d = d > tau ? tau : d;
  }
  // |d| <= tau <= 1 m, so |d 2^20| < 2^31: the 32-bit conversion rounds
  // exactly as a 64-bit one would, and stays off the FP64 pipe
  *dq = (long long)__float2int_rn(__fmul_rn(d, kScale));
  return true;
}

}  // namespace af
