// af_soft.cu -- the differentiable form: soft clearance of (point, direction)
// pairs, its adjoint, fused gradient-ascent refinement, and the SDF views
// they sample.
//
// Soft clearance of a pair (not in the paper; a smooth companion of the tool /
// corridor test of Sec. 3.4): the approach axis from surface point s along
// u = (u0 + alpha t1 + beta t2) / |.| is sampled at a_j = h + j v; sample j
// contributes phi_j = SDF(x_j) - margin_j (tool radius up to the tool length
// L, corridor radius beyond it; samples inside the self-exclusion radius are
// skipped), and C = -tau_s log sum_j exp(-phi_j / tau_s). SDF is trilinear
// interpolation of the TSDF (Sec. 3.2) over voxel centres, tau where
// unobserved.
//
// Views. The hashed map is flattened twice, lazily: all of it on the first
// call, then only the bricks that scans have touched since the last one:
//  * dense : one FP32 SDF per voxel of the map box, row-major (x fastest);
//  * cells : for every interpolation cell (low corner from one voxel below
//            the box to its last voxel) its 8 corner values as two float4,
//            (c000, c100, c010, c110) then (c001, c101, c011, c111), so a
//            sample costs ONE 32-byte sector read. 8x the dense view's size
//            (3.7 GB for a 8 x 8 x 14 m box at 2 cm), traded for sector
//            efficiency -- the memory is there on this part.
//
// Precision. The sample's cell is an integer decided by floating point; it is
// decided in single precision in a fixed order of correctly rounded
// operations (the CPU oracle takes the same decision). The point's position
// is split into its cell I and the offset r in it, so sample positions
// r + (h / v + j) u carry rounding relative to the lever arm, not to the
// distance from the map origin -- which keeps central differences of C in
// single precision meaningful. Interpolation, softmin and gradient use FMA
// and exp2 / log2 freely.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "af_internal.cuh"

namespace af {

// ---------------------------------------------------------------------------
// View builds
// ---------------------------------------------------------------------------

// Bound by the write bandwidth: 16-byte stores from a grid of resident CTAs.
__global__ void __launch_bounds__(256) k_fill(float4* __restrict__ out, size_t n, float value) {
  const float4 v = make_float4(value, value, value, value);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = v;
}

// The pool bricks that a scan has touched since the view last took them: their
// dense SDF (S / (w 2^20) divided in double and rounded to single precision, tau
// where w = 0), and a list of them for k_cell_view. Each scan stamps the hash slot of
// every brick it touches, and `taken` keeps the stamp at which the view took a brick
// (~0: never). Stamps are compared for equality, not order, so scans that run late --
// a captured scan replayed after later ones keeps its older number -- and scan
// numbers that wrap are covered, and a replayed update takes whatever changed
// before it.
//
// A CTA looks at 256 bricks at a time, far apart in the pool (a scan's new bricks
// are neighbours there), and takes each changed one with all its threads: the
// divisions are what a brick costs (a warp to a brick took 2.2 times as long). In a
// small box (`whole`, launch_views) every brick is taken without a look at its
// stamp: the probes and the list would cost more than its few bricks.
__device__ inline void dense_brick(const MapView& M, uint32_t b, float* __restrict__ dense) {
  const size_t X = (size_t)M.dim_vox[0], Y = (size_t)M.dim_vox[1];
  const uint64_t key = M.bkey[b];
  const size_t bx = (size_t)(key & 0x1FFFFF) * 8, by = (size_t)((key >> 21) & 0x1FFFFF) * 8,
               bz = (size_t)(key >> 42) * 8;
  for (int l = threadIdx.x; l < kBrickVox; l += 256) {
    const unsigned long long word = __ldcg(M.vox + (size_t)b * kBrickVox + l);
    const unsigned long long w = word & kWMask;
    const float d = w ? __double2float_rn((double)word_S(word) / ((double)w * 1048576.0)) : M.tau;
    dense[((bz + (l >> 6)) * Y + by + ((l >> 3) & 7)) * X + bx + (l & 7)] = d;
  }
}

__global__ void __launch_bounds__(256) k_dense_view(MapView M, int whole, uint32_t* __restrict__ taken,
                                                    uint32_t* __restrict__ list,
                                                    uint32_t* __restrict__ nlist,
                                                    float* __restrict__ dense) {
  __shared__ uint32_t s_brick[256], s_n, s_first;
  const uint32_t count = min(__ldcg(&M.ctl->pool_count), M.pool_blocks);
  if (whole) {
    for (uint32_t b = blockIdx.x; b < count; b += gridDim.x) dense_brick(M, b, dense);
    return;
  }
  for (uint64_t base = blockIdx.x; base < count; base += 256ull * gridDim.x) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const uint64_t at = base + (uint64_t)threadIdx.x * gridDim.x;
    if (at < count) {
      uint32_t val, stamp;
      if (find_slot(M, M.bkey[at], &val, &stamp) >= 0 && stamp != taken[at]) {
        taken[at] = stamp;
        s_brick[atomicAdd(&s_n, 1u)] = (uint32_t)at;
      }
    }
    __syncthreads();
    const uint32_t n = s_n;
    if (threadIdx.x == 0 && n) s_first = atomicAdd(nlist, n);
    for (uint32_t i = 0; i < n; ++i) dense_brick(M, s_brick[i], dense);
    __syncthreads();
    if (threadIdx.x < n && s_first + threadIdx.x < M.pool_blocks)
      list[s_first + threadIdx.x] = s_brick[threadIdx.x];
    __syncthreads();  // s_brick and s_n are written again
  }
}

// Corner records of the cells that read a voxel of a listed brick: low corners
// from one voxel below the brick to its last voxel, 9^3 cells, from the 10^3
// voxels around it. One CTA per brick, the voxels staged in shared memory, the
// records written in runs of nine (288 bytes). Neighbouring bricks of the list
// write the cells they share twice, with the same values. A block of 8^3 cells
// (cell indices with equal index >> 3) that reads anything but tau is marked in
// `seen`; marks are never cleared (a voxel does not lose its weight). Bound by the record
// writes: a scan of the pine stream changes about 900 bricks, 21 MB of records.
// Rebuilding all 3.7 GB of that box instead took 1.21 ms after each scan; a
// step of scan, scoring and refinement of its 12k points went from 1.56 ms to
// 0.35 ms.
constexpr int kCellEdge = kBrick + 1, kCornerEdge = kBrick + 2;

// The last CTA to end empties the list for the next update (`ended`: zero between
// launches). `whole`: every brick of the box, without a list.
__global__ void __launch_bounds__(256) k_cell_view(MapView M, int whole, const uint32_t* __restrict__ list,
                                                   uint32_t* __restrict__ nlist,
                                                   uint32_t* __restrict__ ended,
                                                   const float* __restrict__ dense,
                                                   float4* __restrict__ cells,
                                                   uint32_t* __restrict__ seen) {
  __shared__ float s_d[kCornerEdge * kCornerEdge * kCornerEdge];
  __shared__ uint32_t s_seen;  // of the 8 blocks the brick's cells lie in
  const int X = M.dim_vox[0], Y = M.dim_vox[1], Z = M.dim_vox[2];
  const uint32_t count = whole ? (uint32_t)((X / 8) * (Y / 8) * (Z / 8)) : min(__ldcg(nlist), M.pool_blocks);
  for (uint32_t k = blockIdx.x; k < count; k += gridDim.x) {
    const uint64_t key = whole ? pack_brick(k % (X / 8), k / (X / 8) % (Y / 8), k / ((X / 8) * (Y / 8)))
                               : M.bkey[list[k]];
    const int bx = (int)(key & 0x1FFFFF) * 8, by = (int)((key >> 21) & 0x1FFFFF) * 8,
              bz = (int)(key >> 42) * 8;
    __syncthreads();  // the previous brick's voxels and marks are no longer read
    if (threadIdx.x == 0) s_seen = 0;
    uint32_t mine = 0;
    for (int i = threadIdx.x; i < kCornerEdge * kCornerEdge * kCornerEdge; i += blockDim.x) {
      const int x = bx - 1 + i % kCornerEdge, y = by - 1 + (i / kCornerEdge) % kCornerEdge,
                z = bz - 1 + i / (kCornerEdge * kCornerEdge);
      const bool in = (unsigned)x < (unsigned)X && (unsigned)y < (unsigned)Y && (unsigned)z < (unsigned)Z;
      s_d[i] = in ? __ldcg(dense + ((size_t)z * Y + y) * X + x) : M.tau;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kCellEdge * kCellEdge * kCellEdge; i += blockDim.x) {
      const int cx = i % kCellEdge, cy = (i / kCellEdge) % kCellEdge, cz = i / (kCellEdge * kCellEdge);
      const float* c = s_d + (cz * kCornerEdge + cy) * kCornerEdge + cx;
      // cell index = low corner + 1 on each axis (the lowest cells lie below the box)
      float4* rec = cells + 2 * (((size_t)(bz + cz) * ((size_t)Y + 1) + (size_t)(by + cy)) * ((size_t)X + 1) +
                                 (size_t)(bx + cx));
      constexpr int sy = kCornerEdge, sz = kCornerEdge * kCornerEdge;
      rec[0] = make_float4(c[0], c[1], c[sy], c[sy + 1]);
      rec[1] = make_float4(c[sz], c[sz + 1], c[sz + sy], c[sz + sy + 1]);
      const float t = M.tau;
      if (c[0] != t || c[1] != t || c[sy] != t || c[sy + 1] != t || c[sz] != t || c[sz + 1] != t ||
          c[sz + sy] != t || c[sz + sy + 1] != t)
        mine |= 1u << ((cx >> 3) | ((cy >> 3) << 1) | ((cz >> 3) << 2));
    }
    mine = __reduce_or_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicOr(&s_seen, mine);
    __syncthreads();
    if (threadIdx.x < 8 && ((s_seen >> threadIdx.x) & 1u)) {
      const size_t b = ((size_t)((bz >> 3) + (threadIdx.x >> 2)) * (Y / 8 + 1) +
                        (size_t)((by >> 3) + ((threadIdx.x >> 1) & 1))) * (X / 8 + 1) +
                       (size_t)((bx >> 3) + (threadIdx.x & 1));
      atomicOr(seen + (b >> 5), 1u << (b & 31));
    }
  }
  if (whole) return;
  __syncthreads();  // every thread has read the count
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ended, 1u) == gridDim.x - 1u) {
      *nlist = 0u;
      *ended = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// Pair geometry, single precision in a fixed order
// ---------------------------------------------------------------------------

// Orthonormal tangent basis (t1, t2) of the unit vector n (Duff et al. 2017,
// "Building an orthonormal basis, revisited").
__device__ inline void onb(const float n[3], float t1[3], float t2[3]) {
  const float sg = n[2] >= 0.0f ? 1.0f : -1.0f;
  const float a = __fdiv_rn(-1.0f, __fadd_rn(sg, n[2]));
  const float b = __fmul_rn(__fmul_rn(n[0], n[1]), a);
  t1[0] = __fadd_rn(1.0f, __fmul_rn(__fmul_rn(__fmul_rn(sg, n[0]), n[0]), a));
  t1[1] = __fmul_rn(sg, b);
  t1[2] = -__fmul_rn(sg, n[0]);
  t2[0] = b;
  t2[1] = __fadd_rn(sg, __fmul_rn(__fmul_rn(n[1], n[1]), a));
  t2[2] = -n[1];
}

// The point's cell on the sample grid (g = x / v - 1/2) and its offset r in
// it, once per pair. `ok` is false for a point whose cell is not a usable
// integer (then every sample reads as outside the view).
struct PointCell {
  float I[3], r[3];
  bool finite, ok;
};

__device__ inline PointCell point_cell(const SoftView& S, const float s[3]) {
  PointCell pc;
  pc.finite = isfinite(s[0]) && isfinite(s[1]) && isfinite(s[2]);
  pc.ok = true;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float o = __fsub_rn(__fdiv_rn(s[i], S.v), 0.5f);
    pc.I[i] = floorf(o);
    pc.r[i] = __fsub_rn(o, pc.I[i]);
    pc.ok = pc.ok && fabsf(pc.I[i]) < 1.0e9f;
  }
  return pc;
}

// The direction of (alpha, beta) around u0 and the standoff in voxels.
struct Dir {
  float u[3];  // unit direction
  float e;     // h / v
  float inq;   // 1 / |u0 + alpha t1 + beta t2|
  bool finite;
};

__device__ inline Dir make_dir(const SoftView& S, const float u0[3], const float t1[3],
                               const float t2[3], float al, float be, float h) {
  Dir d;
  float q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
    q[i] = __fadd_rn(__fadd_rn(u0[i], __fmul_rn(al, t1[i])), __fmul_rn(be, t2[i]));
  const float nq = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(q[0], q[0]), __fmul_rn(q[1], q[1])),
                                        __fmul_rn(q[2], q[2])));
#pragma unroll
  for (int i = 0; i < 3; ++i) d.u[i] = __fdiv_rn(q[i], nq);
  d.e = __fdiv_rn(h, S.v);
  d.inq = 1.0f / nq;
  d.finite = isfinite(al) && isfinite(be) && isfinite(h) && isfinite(u0[0]) &&
             isfinite(u0[1]) && isfinite(u0[2]);
  return d;
}

// Position of the sample at t (standoff plus index, in voxels) in the point's
// cell frame on axis i, in the order of operations the method states.
__device__ inline float sample_pos(const PointCell& pc, const Dir& d, float t, int i) {
  return __fadd_rn(pc.r[i], __fmul_rn(t, d.u[i]));
}

// Where a record is: its index (dense view), or its cell's brick in the brick
// grid and its cell within the brick (sparse view).
template <bool SPARSE>
__device__ inline void record_of(const SoftView& S, const int c[3], uint32_t* idx, uint32_t* loc) {
  if (SPARSE) {
    *idx = ((uint32_t)(c[2] >> 3) * (uint32_t)S.gdim[1] + (uint32_t)(c[1] >> 3)) *
               (uint32_t)S.gdim[0] + (uint32_t)(c[0] >> 3);
    *loc = (uint32_t)((c[0] & 7) | ((c[1] & 7) << 3) | ((c[2] & 7) << 6));
  } else {
    *idx = ((uint32_t)c[2] * (uint32_t)S.ncell[1] + (uint32_t)c[1]) * (uint32_t)S.ncell[0] +
           (uint32_t)c[0];
    *loc = 0;
  }
}

// Cell of the sample at t: false when the cell lies outside the view (all
// corners read tau). f receives the fractional position in the cell.
template <bool SPARSE>
__device__ inline bool sample_cell(const SoftView& S, const PointCell& pc, const Dir& d, float t,
                                   float f[3], int c[3]) {
  bool in = pc.ok;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float l = sample_pos(pc, d, t, i);
    const float fl = floorf(l);
    f[i] = l - fl;  // exact
    const bool ok = fabsf(l) < 1.0e7f;
    const int base = SPARSE ? S.glo[i] : S.lo[i];
    const int lim = SPARSE ? 8 * S.gdim[i] : S.ncell[i];
    c[i] = ok ? (int)pc.I[i] + (int)fl - base : -1;
    in = in && ok && (unsigned)c[i] < (unsigned)lim;
  }
  return in;
}

// The same cell and f for a sample within 2^22 voxels of its point: the floor
// comes from adding 1.5 2^23, which rounds to an integer kept in the low bits --
// four single-precision operations at full rate in the place of a rounding and a
// conversion at a quarter of it. `cb` is the point's cell less the view's base and
// that constant's bits, modulo 2^32 (a point may lie 1e9 cells from the view). Whether the cell lies inside the view is known from the
// sample's index (samples_near).
constexpr float kRound = 12582912.0f;        // 1.5 2^23
constexpr unsigned kRoundBits = 0x4B400000u;
__device__ inline void sample_cell_near(const PointCell& pc, const Dir& d, const unsigned cb[3], float t,
                                        float f[3], int c[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float l = sample_pos(pc, d, t, i);
    const float y0 = __fadd_rn(l, kRound), y = __fsub_rn(y0, kRound);
    const bool up = y > l;  // rounded up: the floor is one below
    f[i] = l - (up ? y - 1.0f : y);
    c[i] = (int)(__float_as_uint(y0) + cb[i] - (up ? 1u : 0u));
  }
}

// Whether every sample j0..J lies within 2^22 voxels of the point and the first
// one inside the view; then the constants of sample_cell_near and the last sample
// inside the view. Rounding is monotone, so on each axis the samples' cells go one
// way: a pair's samples inside the view are the first ones. (Pairs that leave the
// view are ordinary -- every third one where the map box ends half a metre behind
// the surfaces.)
//
// A cell lies inside the view when the sample's position lies between the view's
// faces in the point's frame, whole numbers of cells: two comparisons an axis. (A
// face beyond 2^24 may be rounded; positions within 2^22 compare with it all the
// same.) Where the axis crosses a face is one division for each face that the last
// sample is beyond; the sample before it is then checked, and its neighbours until
// one is inside and the next is not.
template <bool SPARSE>
__device__ inline bool samples_near(const SoftView& S, const PointCell& pc, const Dir& d, unsigned cb[3],
                                    int* last) {
  float face0[3], face1[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const unsigned c0 = (unsigned)(int)pc.I[i] - (unsigned)(SPARSE ? S.glo[i] : S.lo[i]);
    cb[i] = c0 - kRoundBits;
    face0[i] = (float)(int)(0u - c0);
    face1[i] = (float)(int)((unsigned)(SPARSE ? 8 * S.gdim[i] : S.ncell[i]) - c0);
  }
  const auto inside = [&](int j) {
    const float t = __fadd_rn(d.e, (float)j);
    bool in = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float l = sample_pos(pc, d, t, i);
      in = in && l >= face0[i] && l < face1[i];
    }
    return in;
  };
  bool ok = pc.ok, in = true;
  float exit = (float)S.J;  // where the axis leaves the view, in samples
  const float t0 = __fadd_rn(d.e, (float)S.j0), t1 = __fadd_rn(d.e, (float)S.J);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float l0 = sample_pos(pc, d, t0, i), l1 = sample_pos(pc, d, t1, i);
    ok = ok && fabsf(l0) < 4.0e6f && fabsf(l1) < 4.0e6f && l0 >= face0[i] && l0 < face1[i];
    if (l1 < face0[i] || l1 >= face1[i]) {
      in = false;
      exit = fminf(exit, __fdividef((l1 < face0[i] ? face0[i] : face1[i]) - pc.r[i], d.u[i]) - d.e);
    }
  }
  if (!ok) return false;
  int j = S.J;
  if (!in) {
    j = max(S.j0, min(S.J - 1, (int)exit));
    while (j > S.j0 && !inside(j)) --j;
    while (j + 1 < S.J && inside(j + 1)) ++j;
  }
  *last = j;
  return true;
}

__device__ inline float lerp(float a, float b, float t) { return __fmaf_rn(t, b - a, a); }

__device__ inline float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ inline float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Pairs are split across kLanes adjacent lanes: lane g of a pair's group
// takes the samples j0 + g, j0 + g + kLanes, ... and the group merges its
// partial softmin states in a fixed tree onto its first lane, whose result is
// broadcast. Every soft kernel uses the same split, so a pair's C is the same
// bit for bit whichever kernel computes it.
constexpr int kLanes = 4;
constexpr unsigned kFull = 0xffffffffu;

// Softmin state over samples. With FIXED the weights are taken against a
// fixed lower bound `ref` of every phi (no rescaling; the host picks FIXED
// only when the exponents cannot underflow), otherwise against the running
// minimum. m = min phi, Z = sum of exp(-(phi - base) / tau_s), and with GRAD
// the weighted sums sum w_j (h/v + j) G_j and sum w_j G_j of the per-voxel
// SDF gradients G_j.
template <bool GRAD, bool FIXED>
struct Softmin {
  float m = INFINITY, Z = 0.f;
  float at[3] = {0.f, 0.f, 0.f}, a0[3] = {0.f, 0.f, 0.f};

  __device__ inline void scale(float sc) {
    Z *= sc;
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        at[i] *= sc;
        a0[i] *= sc;
      }
    }
  }

  __device__ inline void add(float phi, float t, const float G[3], const SoftView& S) {
    float w;
    if (FIXED) {
      w = ex2((S.ref - phi) * S.k2);
      m = fminf(m, phi);
    } else if (phi < m) {
      scale(ex2((phi - m) * S.k2));
      m = phi;
      w = 1.0f;
    } else {
      w = ex2((m - phi) * S.k2);
    }
    Z += w;
    if (GRAD) {
      const float wt = w * t;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        at[i] = __fmaf_rn(wt, G[i], at[i]);
        a0[i] = __fmaf_rn(w, G[i], a0[i]);
      }
    }
  }

  // this <- this (+) o
  __device__ inline void merge(const Softmin& o, float k2) {
    float sa = 1.f, sb = 1.f;
    const float mm = fminf(m, o.m);
    if (!FIXED) {
      sa = m == INFINITY ? 0.f : ex2((mm - m) * k2);
      sb = o.m == INFINITY ? 0.f : ex2((mm - o.m) * k2);
    }
    Z = Z * sa + o.Z * sb;
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        at[i] = at[i] * sa + o.at[i] * sb;
        a0[i] = a0[i] * sa + o.a0[i] * sb;
      }
    }
    m = mm;
  }

  // Merge the kLanes partial states of the group; every lane gets the result.
  __device__ inline void reduce(float k2) {
#pragma unroll
    for (int off = kLanes / 2; off >= 1; off >>= 1) {
      Softmin o;
      o.m = __shfl_down_sync(kFull, m, off, kLanes);
      o.Z = __shfl_down_sync(kFull, Z, off, kLanes);
      if (GRAD) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          o.at[i] = __shfl_down_sync(kFull, at[i], off, kLanes);
          o.a0[i] = __shfl_down_sync(kFull, a0[i], off, kLanes);
        }
      }
      merge(o, k2);
    }
    m = __shfl_sync(kFull, m, 0, kLanes);
    Z = __shfl_sync(kFull, Z, 0, kLanes);
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        at[i] = __shfl_sync(kFull, at[i], 0, kLanes);
        a0[i] = __shfl_sync(kFull, a0[i], 0, kLanes);
      }
    }
  }
};

// One corner record, 32 bytes, in one 256-bit read-only load.
__device__ inline void load_cell(const SoftView& S, size_t idx, float4& lo, float4& hi) {
  const float4* p = S.cells + 2 * (size_t)idx;
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z),
        "=f"(hi.w)
      : "l"(p));
}

// Trilinear value (and with GRAD its per-voxel gradient) of one record.
template <bool GRAD>
__device__ inline float trilinear(const float4& lo, const float4& hi, const float f[3],
                                  float G[3]) {
  const float dx00 = lo.y - lo.x, dx10 = lo.w - lo.z, dx01 = hi.y - hi.x, dx11 = hi.w - hi.z;
  const float a00 = __fmaf_rn(f[0], dx00, lo.x), a10 = __fmaf_rn(f[0], dx10, lo.z);
  const float a01 = __fmaf_rn(f[0], dx01, hi.x), a11 = __fmaf_rn(f[0], dx11, hi.z);
  const float dy0 = a10 - a00, dy1 = a11 - a01;
  const float b0 = __fmaf_rn(f[1], dy0, a00), b1 = __fmaf_rn(f[1], dy1, a01);
  if (GRAD) {
    G[0] = lerp(lerp(dx00, dx10, f[1]), lerp(dx01, dx11, f[1]), f[2]);
    G[1] = lerp(dy0, dy1, f[2]);
    G[2] = b1 - b0;
  }
  return __fmaf_rn(f[2], b1 - b0, b0);
}

// Records in flight per lane (NF): the lane computes NF sample cells, issues
// their loads, then folds them into the softmin in sample order, so the
// result does not depend on NF. More in flight trade registers for memory
// parallelism: the field of 1.9M pairs takes 487 us with 2, 495 with 3, 545 with
// 4; the refinement of 30k pairs 236 us with 3, 271 with 4 (spills), 263 with 2.
constexpr int kInFlightField = 2;
constexpr int kInFlightRefine = 3;
constexpr int kInFlightRefineFew = 4;  // of few pairs, which wait for latency only
constexpr int kInFlightRefineMid = 3;  // of as many as three CTAs per SM hold
constexpr int kInFlightGeneral = 3;
constexpr int kInFlightGeneralWide = 4;

// Folds lane g's samples j0 + g, j0 + g + kLanes, ... into sm. NEAR: every sample
// lies near the point, those up to `last` inside the view (samples_near); otherwise
// each sample is checked (launch_soft_form says when).
//
// Most samples of a 1.25 m axis read nothing but tau (78% of those of a finished
// pine map), so the dense view's records are only read in blocks of cells that
// hold anything else: one bit per 8^3 cells, 29 KB for the pine box, which stays
// in L1. The records then read are a 27 MB part of the 3.7 GB view and stay in L2.
// With the checks of the cells gone as well, the field of a finished map's 30k
// points (1.9M pairs) went from 862 to about 485 us, forward plus adjoint of 113k
// pairs from 149 to 71 us, the refinement of 30k pairs from 315 to 232 us. In a
// small box (0.17 GB of records, which the caches hold) they gain nothing: 512k
// pairs, a third of which leave the view, take 127 us either way.
template <bool NEAR, bool GRAD, bool FIXED, bool SPARSE, int NF>
__device__ inline void fold_samples(Softmin<GRAD, FIXED>& sm, const SoftView& S, const PointCell& pc,
                                    const Dir& d, const unsigned cb[3], int last, int g) {
#pragma unroll 1
  for (int j = S.j0 + g; j <= S.J; j += NF * kLanes) {
    float f[NF][3];
    uint32_t id[NF], loc[NF];
    size_t rec[NF];
    bool has[NF], in[NF];
    uint32_t mark[NF], bit[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) {
      has[q] = j + q * kLanes <= S.J;
      const float t = __fadd_rn(d.e, (float)(j + q * kLanes));
      int c[3];
      if (NEAR) {
        sample_cell_near(pc, d, cb, t, f[q], c);
        in[q] = j + q * kLanes <= last;
      } else {
        in[q] = has[q] && sample_cell<SPARSE>(S, pc, d, t, f[q], c);
      }
      record_of<SPARSE>(S, c, &id[q], &loc[q]);
      rec[q] = id[q];
      if (!SPARSE && NEAR) {
        const uint32_t b = ((uint32_t)(c[2] >> 3) * (uint32_t)S.nblock[1] + (uint32_t)(c[1] >> 3)) *
                               (uint32_t)S.nblock[0] + (uint32_t)(c[0] >> 3);
        mark[q] = in[q] ? __ldg(S.seen + (b >> 5)) : 0u;
        bit[q] = b;
      }
    }
    if (SPARSE) {  // the slots of the cells' bricks first, then the records
      uint32_t slot[NF];
#pragma unroll
      for (int q = 0; q < NF; ++q) slot[q] = in[q] ? __ldg(S.bgrid + id[q]) : kNoBlock;
#pragma unroll
      for (int q = 0; q < NF; ++q) {
        in[q] = in[q] && slot[q] != kNoBlock;
        rec[q] = (size_t)slot[q] * kBrickVox + loc[q];
      }
    } else if (NEAR) {
#pragma unroll
      for (int q = 0; q < NF; ++q) in[q] = (mark[q] >> (bit[q] & 31u)) & 1u;
    }
    float4 lo[NF], hi[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q)
      if (in[q]) load_cell(S, rec[q], lo[q], hi[q]);
#pragma unroll
    for (int q = 0; q < NF; ++q) {
      if (!has[q]) break;
      const int jq = j + q * kLanes;
      float G[3] = {0.f, 0.f, 0.f};
      const float D = in[q] ? trilinear<GRAD>(lo[q], hi[q], f[q], G) : S.tau;
      sm.add(D - (jq <= S.jt ? S.r : S.r_corr), d.e + (float)jq, G, S);
    }
  }
}

// How a kernel takes its samples: the short way for every pair whose samples lie
// near its point and the general way for the others (kBoth), the others not at all
// (kNear: *far is set instead), every pair the general way (kGeneral; kRedo: those
// that a kNear launch has left).
enum Road { kBoth, kNear, kGeneral, kRedo };

// C of one pair and, with GRAD, dC / d(alpha, beta, h); *cmin = min_j phi_j.
// Called by all kLanes lanes of the pair's group (lane g of it); with
// `live` false the lane samples nothing.
template <bool GRAD, bool FIXED, bool SPARSE, int NF, Road ROAD>
__device__ inline float soft_eval(const SoftView& S, const PointCell& pc, const Dir& d,
                                  const float t1[3], const float t2[3], bool live, int g,
                                  float* ga, float* gb, float* gh, float* cmin, bool* far) {
  Softmin<GRAD, FIXED> sm;
  if (live) {
    unsigned cb[3] = {0u, 0u, 0u};
    int last = 0;
    if ((ROAD == kBoth || ROAD == kNear) && samples_near<SPARSE>(S, pc, d, cb, &last))
      fold_samples<true, GRAD, FIXED, SPARSE, NF>(sm, S, pc, d, cb, last, g);
    else if (ROAD == kNear)
      *far = true;
    else
      fold_samples<false, GRAD, FIXED, SPARSE, ROAD == kBoth ? 1 : NF>(sm, S, pc, d, cb, 0, g);
  }
  sm.reduce(S.k2);
  const float C = (FIXED ? S.ref : sm.m) - S.ln2_tau_s * lg2(sm.Z);
  *cmin = sm.m;
  if (GRAD) {
    // du/dalpha = (t1 - u (u . t1)) / |q|, likewise for beta with t2
    const float iz = 1.0f / sm.Z;
    const float au = sm.at[0] * d.u[0] + sm.at[1] * d.u[1] + sm.at[2] * d.u[2];
    const float ut1 = d.u[0] * t1[0] + d.u[1] * t1[1] + d.u[2] * t1[2];
    const float ut2 = d.u[0] * t2[0] + d.u[1] * t2[1] + d.u[2] * t2[2];
    const float at1 = sm.at[0] * t1[0] + sm.at[1] * t1[1] + sm.at[2] * t1[2];
    const float at2 = sm.at[0] * t2[0] + sm.at[1] * t2[1] + sm.at[2] * t2[2];
    *ga = (at1 - au * ut1) * d.inq * iz;
    *gb = (at2 - au * ut2) * d.inq * iz;
    *gh = (sm.a0[0] * d.u[0] + sm.a0[1] * d.u[1] + sm.a0[2] * d.u[2]) * iz / S.v;
  }
  return C;
}

__device__ inline void load3(const float* __restrict__ p, size_t i, float o[3]) {
  o[0] = __ldg(p + 3 * i);
  o[1] = __ldg(p + 3 * i + 1);
  o[2] = __ldg(p + 3 * i + 2);
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_soft_seed(const float* __restrict__ nrm, uint32_t m,
                                                   const float* __restrict__ table, uint32_t K,
                                                   float* __restrict__ u0) {
  const size_t n = (size_t)m * K;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    float nv[3], e[3], t1[3], t2[3];
    load3(nrm, i / K, nv);
    load3(table, i % K, e);
    onb(nv, t1, t2);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      u0[3 * i + k] = __fadd_rn(__fadd_rn(__fmul_rn(e[0], t1[k]), __fmul_rn(e[1], t2[k])),
                                __fmul_rn(e[2], nv[k]));
  }
}

// Pair groups of a warp, walked so that every lane of the warp takes the same
// number of iterations (the group merges are warp-wide shuffles).
struct GroupWalk {
  size_t first, stride;
  int g, slot;
  __device__ GroupWalk() {
    const int lane = threadIdx.x & 31;
    g = lane % kLanes;
    slot = lane / kLanes;
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    first = warp * (32 / kLanes);
    stride = warps * (32 / kLanes);
  }
};

template <bool GRAD, bool FIXED, bool SPARSE, Road ROAD, int NF>
__global__ void __launch_bounds__(128) k_soft(SoftView S, const float* __restrict__ pts,
                                              uint32_t per_point, const float* __restrict__ u0,
                                              const float* __restrict__ alpha,
                                              const float* __restrict__ beta,
                                              const float* __restrict__ hh, uint64_t n,
                                              const float* __restrict__ gc, float* __restrict__ c,
                                              float* __restrict__ cmin, float* __restrict__ ga,
                                              float* __restrict__ gb, float* __restrict__ gh) {
  const GroupWalk w;
  for (size_t base = w.first; base < n; base += w.stride) {
    const size_t i0 = base + w.slot;
    const bool act = i0 < n;
    const size_t i = act ? i0 : n - 1;
    float s[3], u[3], t1[3], t2[3];
    load3(pts, i / per_point, s);
    load3(u0, i, u);
    onb(u, t1, t2);
    const PointCell pc = point_cell(S, s);
    const Dir d = make_dir(S, u, t1, t2, __ldg(alpha + i), __ldg(beta + i), __ldg(hh + i));
    const bool fin = pc.finite && d.finite;
    float da, db, dh, mn;
    float C = soft_eval<GRAD, FIXED, SPARSE, NF, ROAD>(S, pc, d, t1, t2, fin && act, w.g, &da, &db, &dh,
                                                       &mn, nullptr);
    if (!act || w.g != 0) continue;
    if (!fin) C = mn = da = db = dh = NAN;
    if (c) c[i] = C;
    if (cmin) cmin[i] = mn;
    if (GRAD) {
      const float gg = gc ? __ldg(gc + i) : 1.0f;
      if (ga) ga[i] = gg * da;
      if (gb) gb[i] = gg * db;
      if (gh) gh[i] = gg * dh;
    }
  }
}

// `steps` ascent steps on C of pair i in registers, then C at the final state;
// the group's lanes (`act`: the pair is taken) update identical copies of
// (alpha, beta, h). False, with nothing written, if a step takes a sample far from
// the point (ROAD == kNear).
template <bool FIXED, bool SPARSE, int NF, Road ROAD>
__device__ inline bool refine_pair(const SoftView& S, const RefineArgs& R, const float* __restrict__ pts,
                                   uint32_t per_point, const float* __restrict__ u0,
                                   float* __restrict__ alpha, float* __restrict__ beta,
                                   float* __restrict__ hh, float* __restrict__ c,
                                   float* __restrict__ cmin, size_t i, bool act, int g) {
  float s[3], u[3], t1[3], t2[3];
  load3(pts, i / per_point, s);
  load3(u0, i, u);
  onb(u, t1, t2);
  const PointCell pc = point_cell(S, s);
  float al = alpha[i], be = beta[i], h = hh[i];
  // a pair that is not finite (e.g. a point with no start) samples nothing
  const bool fin = pc.finite && make_dir(S, u, t1, t2, al, be, h).finite;
  bool far = false;
#pragma unroll 1
  for (int k = 0; k < R.steps; ++k) {
    const Dir d = make_dir(S, u, t1, t2, al, be, h);
    const bool live = fin && act && d.finite && !far;
    float da, db, dh, mn;
    soft_eval<true, FIXED, SPARSE, NF, ROAD>(S, pc, d, t1, t2, live, g, &da, &db, &dh, &mn, &far);
    if (live) {
      al = __fmaf_rn(R.lr_dir, da, al);
      be = __fmaf_rn(R.lr_dir, db, be);
      h = fminf(fmaxf(__fmaf_rn(R.lr_h, dh, h), 0.0f), R.h_max);
    }
  }
  const Dir d = make_dir(S, u, t1, t2, al, be, h);
  const bool ok = fin && d.finite;
  float mn;
  float C = soft_eval<false, FIXED, SPARSE, NF, ROAD>(S, pc, d, t1, t2, ok && act && !far, g, nullptr,
                                                      nullptr, nullptr, &mn, &far);
  if (!act || far || g != 0) return !far;
  if (!ok) C = mn = al = be = h = NAN;
  alpha[i] = al;
  beta[i] = be;
  hh[i] = h;
  c[i] = C;
  if (cmin) cmin[i] = mn;
  return true;
}

// Two launches: the general way beside the short one would cost every pair 70
// registers, so the first (ROAD kNear) leaves a pair that it cannot take
// (samples_near) as it was and marks its C with a NaN of its own, and the second
// takes the marked pairs from their start again.
constexpr unsigned kRedoMark = 0x7FC05EDDu;

template <bool FIXED, bool SPARSE, Road ROAD, int NF, int CTAS>
__global__ void __launch_bounds__(128, CTAS) k_soft_refine(SoftView S, RefineArgs R,
                                                     const float* __restrict__ pts,
                                                     uint32_t per_point,
                                                     const float* __restrict__ u0,
                                                     float* __restrict__ alpha,
                                                     float* __restrict__ beta,
                                                     float* __restrict__ hh, uint64_t n,
                                                     float* __restrict__ c,
                                                     float* __restrict__ cmin) {
  const GroupWalk w;
  for (size_t base = w.first; base < n; base += w.stride) {
    const size_t i0 = base + w.slot;
    bool act = i0 < n;
    const size_t i = act ? i0 : n - 1;
    if (ROAD == kRedo) {
      act = act && __float_as_uint(c[i]) == kRedoMark;
      if (!__any_sync(kFull, act)) continue;
    }
    if (!refine_pair<FIXED, SPARSE, NF, ROAD>(
            S, R, pts, per_point, u0, alpha, beta, hh, c, cmin, i, act, w.g) && act && w.g == 0)
      c[i] = __uint_as_float(kRedoMark);
  }
}

// Start of each point's refinement from the plain path's result: the best
// direction of an ACCESSIBLE point, NaN otherwise (refinement skips it).
__global__ void __launch_bounds__(256) k_soft_start(const uint8_t* __restrict__ label,
                                                    const int16_t* __restrict__ best, uint32_t m,
                                                    const float* __restrict__ dirs, int G,
                                                    float* __restrict__ u0) {
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < m; p += gridDim.x * blockDim.x) {
    const int b = best[p];
    const bool ok = label[p] == 1 && b >= 0 && b < G;
#pragma unroll
    for (int d = 0; d < 3; ++d) u0[3 * p + d] = ok ? __ldg(dirs + 3 * b + d) : NAN;
  }
}

// Per point: the index (within the point's pairs) and value of the largest C,
// lowest index on ties, -1 when every C is NaN; optionally that pair's base
// direction (NaN for -1).
__global__ void __launch_bounds__(256) k_soft_best(const float* __restrict__ c, uint64_t n,
                                                   uint32_t per_point, uint64_t points,
                                                   const float* __restrict__ u0,
                                                   int32_t* __restrict__ best_k,
                                                   float* __restrict__ best_c,
                                                   float* __restrict__ best_u0) {
  for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < points;
       p += (size_t)gridDim.x * blockDim.x) {
    const size_t a = p * per_point, b = min((size_t)n, a + per_point);
    int32_t k = -1;
    float v = NAN;
    for (size_t i = a; i < b; ++i) {
      const float x = c[i];
      if (x == x && (k < 0 || x > v)) {
        k = (int32_t)(i - a);
        v = x;
      }
    }
    if (best_k) best_k[p] = k;
    if (best_c) best_c[p] = v;
    if (best_u0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) best_u0[3 * p + d] = k >= 0 ? u0[3 * (a + k) + d] : NAN;
    }
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------

static unsigned grid_for(size_t n, int threads, int num_sms, int per_sm) {
  const size_t want = (n + threads - 1) / threads;
  const size_t cap = (size_t)num_sms * per_sm;
  return (unsigned)(want < cap ? (want ? want : 1) : cap);
}

// ---- the brick-sparse view ----
//
// A cell (low corner c, corners c + {0,1}^3) has corners in the bricks of c
// and the ones above it on each axis, so a cell with a corner in an
// allocated brick B has its low corner in B - e for some e in {0,1}^3; every
// other cell reads tau at all corners. The grid covers the box's bricks and
// one layer below (cells whose low corner lies one voxel below the box);
// each brick of {B - e} gets a slot of 512 corner records, the others none.

// Marks every grid brick B - e (B allocated, e in {0,1}^3) with a slot; one
// thread per (allocated brick, e).
__global__ void __launch_bounds__(256) k_sview_mark(MapView M, uint32_t* __restrict__ bgrid,
                                                    int gx, int gy, uint32_t* __restrict__ keys,
                                                    uint32_t* __restrict__ nslots) {
  const uint32_t count = min(__ldcg(&M.ctl->pool_count), M.pool_blocks);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count * 8u;
       i += gridDim.x * blockDim.x) {
    const uint64_t key = M.bkey[i >> 3];
    const int e = (int)(i & 7u);
    // grid coordinates: box-relative brick + 1 (the layer below the box is 0)
    const int x = (int)(key & 0x1FFFFF) + 1 - (e & 1), y = (int)((key >> 21) & 0x1FFFFF) + 1 - ((e >> 1) & 1),
              z = (int)(key >> 42) + 1 - (e >> 2);
    const uint32_t t = ((uint32_t)z * (uint32_t)gy + (uint32_t)y) * (uint32_t)gx + (uint32_t)x;
    if (atomicCAS(bgrid + t, kNoBlock, kNoBlock - 1u) == kNoBlock) {
      const uint32_t s = atomicAdd(nslots, 1u);
      keys[s] = t;
      bgrid[t] = s;
    }
  }
}

// The 512 corner records of every slot: one CTA of 512 threads per slot, the
// pool indices of the 8 bricks its cells' corners can lie in looked up once.
__global__ void __launch_bounds__(512) k_sview_fill(MapView M, const uint32_t* __restrict__ keys,
                                                    uint32_t nslots, int gx, int gy,
                                                    float4* __restrict__ cells) {
  __shared__ uint32_t s_nb[8];
  const int l = threadIdx.x;
  const int X = M.dim_vox[0], Y = M.dim_vox[1], Z = M.dim_vox[2];
  for (uint32_t s = blockIdx.x; s < nslots; s += gridDim.x) {
    const uint32_t t = keys[s];
    // box-relative brick of the slot's low corners
    const int bx = (int)(t % (uint32_t)gx) - 1, by = (int)((t / (uint32_t)gx) % (uint32_t)gy) - 1,
              bz = (int)(t / ((uint32_t)gx * (uint32_t)gy)) - 1;
    __syncthreads();  // s_nb of the previous slot is no longer read
    if (l < 8) {
      const int x = bx + (l & 1), y = by + ((l >> 1) & 1), z = bz + (l >> 2);
      s_nb[l] = (x >= 0 && y >= 0 && z >= 0 && x * 8 < X && y * 8 < Y && z * 8 < Z)
                    ? lookup_brick(M, pack_brick(x, y, z))
                    : kNoBlock;
    }
    __syncthreads();
    const int vx = bx * 8 + (l & 7), vy = by * 8 + ((l >> 3) & 7), vz = bz * 8 + (l >> 6);
    float c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int x = vx + (k & 1), y = vy + ((k >> 1) & 1), z = vz + (k >> 2);
      float d = M.tau;  // outside the box, unallocated, or w = 0
      if (x >= 0 && y >= 0 && z >= 0 && x < X && y < Y && z < Z) {
        const uint32_t b = s_nb[((x >> 3) - bx) | (((y >> 3) - by) << 1) | (((z >> 3) - bz) << 2)];
        if (b != kNoBlock) {
          const unsigned long long word =
              __ldcg(M.vox + (size_t)b * kBrickVox + ((x & 7) | ((y & 7) << 3) | ((z & 7) << 6)));
          const unsigned long long w = word & kWMask;
          if (w) d = __double2float_rn((double)word_S(word) / ((double)w * 1048576.0));
        }
      }
      c[k] = d;
    }
    float4* rec = cells + 2 * ((size_t)s * kBrickVox + l);
    rec[0] = make_float4(c[0], c[1], c[2], c[3]);
    rec[1] = make_float4(c[4], c[5], c[6], c[7]);
  }
}

cudaError_t launch_sview_mark(const MapView& M, int num_sms, uint32_t* bgrid, size_t gcount,
                              int gx, int gy, uint32_t* keys, uint32_t* nslots, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(bgrid, 0xFF, gcount * 4, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(nslots, 0, 4, stream);
  if (e != cudaSuccess) return e;
  k_sview_mark<<<num_sms * 8, 256, 0, stream>>>(M, bgrid, gx, gy, keys, nslots);
  return cudaGetLastError();
}

cudaError_t launch_sview_fill(const MapView& M, int num_sms, const uint32_t* keys, uint32_t nslots,
                              int gx, int gy, float4* cells, cudaStream_t stream) {
  if (nslots == 0) return cudaSuccess;
  k_sview_fill<<<(unsigned)std::min<uint32_t>(nslots, (uint32_t)num_sms * 4), 512, 0, stream>>>(
      M, keys, nslots, gx, gy, cells);
  return cudaGetLastError();
}

// Words of the dense view's list: the bricks of an update, their count, its ended
// CTAs, and the stamp at which the view took each brick.
size_t view_list_words(const MapView& M) { return 2 * (size_t)M.pool_blocks + 2; }

// Words of the dense view's block marks.
size_t seen_words(const MapView& M) {
  const size_t n = ((size_t)M.dim_vox[0] / 8 + 1) * (M.dim_vox[1] / 8 + 1) * (M.dim_vox[2] / 8 + 1);
  return (n + 31) / 32;
}

// Brings the dense view up to date with the map; with `fill` the buffers are new,
// every value starts as tau and every brick is taken. `list`: view_list_words(M).
// *kernels: the kernels launched.
cudaError_t launch_views(const MapView& M, int num_sms, bool fill, float* dense, float4* cells,
                         uint32_t* list, uint32_t* seen, int* kernels, cudaStream_t stream) {
  *kernels = fill ? 4 : 2;
  const size_t nd = (size_t)M.dim_vox[0] * M.dim_vox[1] * M.dim_vox[2];  // a multiple of 512
  const size_t nc = ((size_t)M.dim_vox[0] + 1) * (M.dim_vox[1] + 1) * (M.dim_vox[2] + 1);
  uint32_t *nlist = list + M.pool_blocks, *ended = nlist + 1, *taken = nlist + 2;
  if (fill) {
    k_fill<<<grid_for(nd / 4, 256, num_sms, 8), 256, 0, stream>>>(reinterpret_cast<float4*>(dense),
                                                                   nd / 4, M.tau);
    k_fill<<<grid_for(nc * 2, 256, num_sms, 8), 256, 0, stream>>>(cells, nc * 2, M.tau);
    cudaError_t z = cudaMemsetAsync(seen, 0, seen_words(M) * sizeof(uint32_t), stream);
    if (z == cudaSuccess) z = cudaMemsetAsync(nlist, 0, 2 * sizeof(uint32_t), stream);
    if (z == cudaSuccess) z = cudaMemsetAsync(taken, 0xFF, M.pool_blocks * sizeof(uint32_t), stream);
    if (z != cudaSuccess) return z;
  }
  // A CTA for each brick that there can be, up to a chip full of them. Boxes of up to
  // four bricks per SM are taken whole: 8^3 bricks 20 us a scan, by their stamps 22 (26
  // with the list in a launch of its own and a memset); 12^3 bricks by stamps 21, whole 25.
  const size_t bricks = nd / kBrickVox;
  const int whole = bricks <= (size_t)num_sms * 4;
  const unsigned grid = (unsigned)std::min<size_t>(bricks, (size_t)num_sms * 8);
  k_dense_view<<<grid, 256, 0, stream>>>(M, whole, taken, list, nlist, dense);
  k_cell_view<<<grid, 256, 0, stream>>>(M, whole, list, nlist, ended, dense, cells, seen);
  return cudaGetLastError();
}

cudaError_t launch_soft_seed(const float* d_nrm, uint32_t m, const float* d_table, uint32_t K,
                             float* d_u0, int num_sms, cudaStream_t stream) {
  const size_t n = (size_t)m * K;
  if (n == 0) return cudaSuccess;
  k_soft_seed<<<grid_for(n, 256, num_sms, 8), 256, 0, stream>>>(d_nrm, m, d_table, K, d_u0);
  return cudaGetLastError();
}

// Which way the samples go, by their number per pair. The short way costs each
// evaluation about as much as four samples a lane (the view's faces, the last
// sample inside) and spares a quarter of each sample's work, so few samples go the
// general way. In a box whose records the caches hold the marks spare nothing as
// well, and the line lies higher; without marks (sparse view) it lies lower, since
// the general way has a slot to read for every sample. Field of 512k pairs with 8 / 12
// / 20 / 28 / 36 / 62 samples, short against general way: in the pine's dense view
// 49 / 59 / 74 / 88 / 102 / 137 us against 45 / 49 / 67 / 94 / 119 / 243; in a box of
// 0.17 GB of records 49 / 59 / 70 / 81 / 92 / 127 against 46 / 50 / 63 / 77 / 86 / 127;
// in the sparse view 50 / 61 / 77 / 93 / 108 / 153 against 51 / 58 / 78 / 97 / 110 / 160.
constexpr int kGeneralBelow = 25, kGeneralBelowSmallBox = 49, kGeneralBelowSparse = 17;
constexpr uint64_t kSmallBoxCells = 1ull << 23;  // 0.25 GB of records

template <bool GRAD, bool FIXED, bool SPARSE>
static void launch_soft_form(const SoftView& S, const float* pts, uint32_t per_point, const float* u0,
                             const float* al, const float* be, const float* h, uint64_t n,
                             const float* gc, float* c, float* cmin, float* ga, float* gb, float* gh,
                             int num_sms, cudaStream_t stream) {
  const int samples = S.J - S.j0 + 1;
  const bool small = (uint64_t)S.ncell[0] * S.ncell[1] * S.ncell[2] <= kSmallBoxCells;
  const unsigned g = grid_for(n * kLanes, 128, num_sms, 16);
  const auto run = [&](auto kernel) {
    kernel<<<g, 128, 0, stream>>>(S, pts, per_point, u0, al, be, h, n, gc, c, cmin, ga, gb, gh);
  };
  if (samples < (SPARSE ? kGeneralBelowSparse : small ? kGeneralBelowSmallBox : kGeneralBelow))
    run(k_soft<GRAD, FIXED, SPARSE, kGeneral, kInFlightGeneral>);
  else
    run(k_soft<GRAD, FIXED, SPARSE, kBoth, kInFlightField>);
}

cudaError_t launch_soft(const SoftView& S, bool grad, const float* pts, uint32_t per_point,
                        const float* u0, const float* al, const float* be, const float* h,
                        uint64_t n, const float* gc, float* c, float* cmin, float* ga,
                        float* gb, float* gh, int num_sms, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  decltype(&launch_soft_form<false, false, false>) form =
      grad ? (S.fixed ? (S.sparse ? launch_soft_form<true, true, true> : launch_soft_form<true, true, false>)
                      : (S.sparse ? launch_soft_form<true, false, true> : launch_soft_form<true, false, false>))
           : (S.fixed ? (S.sparse ? launch_soft_form<false, true, true> : launch_soft_form<false, true, false>)
                      : (S.sparse ? launch_soft_form<false, false, true>
                                  : launch_soft_form<false, false, false>));
  form(S, pts, per_point, u0, al, be, h, n, gc, c, cmin, ga, gb, gh, num_sms, stream);
  return cudaGetLastError();
}

// Refinement, by the samples per pair as above (its evaluations carry gradients, so
// a sample spared counts for more) and by how many pairs the chip holds at once.
//  * Few samples: the general way, four records in flight and three CTAs per SM, or
//    three and four where that takes a wave less. 14k pairs with 8 / 12 / 20 samples:
//    47 / 52 / 67 us, the short way in two launches 56 / 60 / 74; 15k pairs 52 / 57 /
//    74, in two waves of three CTAs 69 / 75 / 99.
//  * In the dense view up to 32 samples, two rounds of four a lane: the same, if it
//    takes no wave more and the pairs are more than the next form holds (10k pairs
//    with 28 samples 69 against 80 us).
//  * As many pairs as two CTAs per SM hold: latency is all that counts, four records
//    in flight, both ways in one kernel (220 registers).
//  * As many as three CTAs per SM hold: both ways in one kernel of three records
//    in flight (12k pairs of a small box with 62 samples 109 us, in two launches 113).
//  * More: the short way in four CTAs per SM, and a second launch for what it left
//    (25k pairs on the pine map 219 us).
constexpr int kRefineGeneralBelow = 25, kRefineGeneralBelowSparse = 9, kRefineWideBelow = 33;

template <bool FIXED, bool SPARSE>
static void launch_refine_form(const SoftView& S, const RefineArgs& R, const float* pts,
                               uint32_t per_point, const float* u0, float* al, float* be, float* h,
                               uint64_t n, float* c, float* cmin, int num_sms, int* kernels,
                               cudaStream_t stream) {
  const int samples = S.J - S.j0 + 1;
  const unsigned g = grid_for(n * kLanes, 128, num_sms, 16);
  const auto waves = [&](int ctas) {
    const uint64_t held = (uint64_t)num_sms * ctas * (128 / kLanes);
    return (n + held - 1) / held;
  };
  const auto run = [&](auto kernel) {
    kernel<<<g, 128, 0, stream>>>(S, R, pts, per_point, u0, al, be, h, n, c, cmin);
    ++*kernels;
  };
  const int few_samples = SPARSE ? kRefineGeneralBelowSparse : kRefineGeneralBelow;
  const bool wide = waves(3) == waves(4);
  if (samples < few_samples && !wide) {
    run(k_soft_refine<FIXED, SPARSE, kGeneral, kInFlightGeneral, 4>);
  } else if (wide && (samples < few_samples ||
                      (!SPARSE && samples < kRefineWideBelow && waves(2) > 1))) {
    run(k_soft_refine<FIXED, SPARSE, kGeneral, kInFlightGeneralWide, 3>);
  } else if (waves(2) == 1) {
    run(k_soft_refine<FIXED, SPARSE, kBoth, kInFlightRefineFew, 2>);
  } else if (waves(3) == 1) {
    run(k_soft_refine<FIXED, SPARSE, kBoth, kInFlightRefineMid, 3>);
  } else {
    run(k_soft_refine<FIXED, SPARSE, kNear, kInFlightRefine, 4>);
    run(k_soft_refine<FIXED, SPARSE, kRedo, 1, 4>);
  }
}

cudaError_t launch_soft_refine(const SoftView& S, const RefineArgs& R, const float* pts,
                               uint32_t per_point, const float* u0, float* al, float* be,
                               float* h, uint64_t n, float* c, float* cmin, int num_sms,
                               int* kernels, cudaStream_t stream) {
  *kernels = 0;
  if (n == 0) return cudaSuccess;
  decltype(&launch_refine_form<false, false>) form =
      S.fixed ? (S.sparse ? launch_refine_form<true, true> : launch_refine_form<true, false>)
              : (S.sparse ? launch_refine_form<false, true> : launch_refine_form<false, false>);
  form(S, R, pts, per_point, u0, al, be, h, n, c, cmin, num_sms, kernels, stream);
  return cudaGetLastError();
}

cudaError_t launch_soft_start(const uint8_t* label, const int16_t* best, uint32_t m,
                              const float* dirs, int G, float* u0, int num_sms,
                              cudaStream_t stream) {
  if (m == 0) return cudaSuccess;
  k_soft_start<<<grid_for(m, 256, num_sms, 8), 256, 0, stream>>>(label, best, m, dirs, G, u0);
  return cudaGetLastError();
}

cudaError_t launch_soft_best(const float* c, uint64_t n, uint32_t per_point, const float* u0,
                             int32_t* best_k, float* best_c, float* best_u0, int num_sms,
                             cudaStream_t stream) {
  const uint64_t points = (n + per_point - 1) / per_point;
  if (points == 0) return cudaSuccess;
  k_soft_best<<<grid_for(points, 256, num_sms, 8), 256, 0, stream>>>(c, n, per_point, points, u0,
                                                                      best_k, best_c, best_u0);
  return cudaGetLastError();
}

}  // namespace af
