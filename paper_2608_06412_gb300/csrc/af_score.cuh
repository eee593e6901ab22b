// af_score.cuh -- the scoring device functions (Sec. 3.4, 3.5), shared by the
// plain, batched and stateful-layer scoring kernels.
//
// Kernels are quads rather than voxel lists. The views keep the 32-bit words of
// a 2 x 2 group of rows side by side (af_internal.cuh), so one 16-byte load
// reads 32 voxels of four neighbouring rows. A kernel's voxels are grouped the
// same way: an entry is a group of rows (as an offset from the point's group),
// a window of up to 32 voxels along the rows' axis and one mask per row. Which
// voxels share a group depends on the parity of the point's coordinates across
// the axis, so each direction has its entries four times, once per parity; the
// position along the axis is free (a funnel shift of the two words the window
// may straddle). Each direction follows the axis it is closest to, read from
// the occupied view with rows along that axis.
//
// Why quads: the search of a point is a chain of dependent loads, one warp step
// each, and off-axis kernels cut rows into short runs (7 voxels on average for
// the 1 m corridor at 2 cm). Per direction of the 4 cm tool a run each row takes
// 32 tool and 143 corridor loads, quads about 12 and 47: a tool fits 8 or 16
// lanes, so four directions are counted side by side, and a corridor is walked
// in two steps instead of five. Against runs with their tables staged in
// shared memory: 72.5 -> 53 us per pine frame (12k points, 128 directions), 489
// -> 282 us for 40k points of three pines with the 6 cm tool and 256 directions,
// 2.5 -> 1.28 ms for 83k points of a 1 cm map with 512. The latter two are bound
// by L1 wavefronts (82% of their peak on the 1 cm map: a gather of 16-byte words
// takes a wavefront per lane), the pine frame by the chain and its tail.
//
// A point whose whole kernel reach lies inside the map box takes the FAST path,
// which checks no bound; otherwise words outside the box read as zero: nothing
// occupied, nothing known.
#pragma once

#include "af_internal.cuh"

namespace af {

struct Pt {
  int px, py, pz;  // box-relative voxel of the point
};

// Whether every voxel that any kernel or arm sample reaches from P lies inside
// the map box.
__device__ __forceinline__ bool reach_inside(const MapView& M, const ToolView& T, const Pt& P) {
  return P.px >= T.reach[0] && P.px + T.reach[0] < M.dim_vox[0] && P.py >= T.reach[1] &&
         P.py + T.reach[1] < M.dim_vox[1] && P.pz >= T.reach[2] && P.pz + T.reach[2] < M.dim_vox[2];
}

// A direction's entries as seen from a point: tool entries [t0, t0 + nt) and
// corridor entries [c0, c0 + nc) of the point's parity, the axis of its rows,
// and the point's place on the view with rows along that axis.
struct DirRows {
  int t0, nt, c0, nc;
  const uint4* view;
  int axis;
  int a, o1, o2;  // the point's coordinates: along the rows, and the other two (o1 the lower axis)
};

// Parity of the point's row group: which copy of a direction's entries applies.
__device__ __forceinline__ int parity(int o1, int o2) { return (o1 & 1) | ((o2 & 1) << 1); }

// `d`: the direction's table entry. `along_x`: its corridor entries follow x
// (strict) whatever the direction's axis.
__device__ __forceinline__ DirRows dir_rows(const MapView& M, const Pt& P, int4 d, bool along_x = false) {
  DirRows r;
  r.axis = along_x ? 0 : (int)((uint32_t)d.x >> kAxisShift);
  r.view = r.axis == 0 ? M.occ : (r.axis == 1 ? M.occ_y : M.occ_z);
  r.a = r.axis == 0 ? P.px : (r.axis == 1 ? P.py : P.pz);
  r.o1 = r.axis == 0 ? P.py : P.px;
  r.o2 = r.axis == 2 ? P.py : P.pz;
  r.nt = d.y;
  r.nc = d.w;
  r.t0 = (d.x & kEntryMask) + parity(r.o1, r.o2) * d.y;
  r.c0 = d.z + parity(r.o1, r.o2) * d.w;
  return r;
}

// The masked bits of entry i (four rows) seen from D's point on `view`.
template <bool FAST>
__device__ __forceinline__ uint4 quad_bits(const MapView& M, const ToolView& T, const DirRows& D,
                                           const uint4* __restrict__ view, int i, uint4* mask) {
  if (!check_index((unsigned)i < (unsigned)T.nent, M.ctl)) {
    *mask = make_uint4(0u, 0u, 0u, 0u);
    return *mask;
  }
  const int2 e = __ldg(T.qent + i);  // (group offsets q1 | q2 << 16, d0 << 16 | 32 - window)
  const uint4 m = __ldg(T.qmask + i);
  *mask = m;
  const int xa = D.a + (e.y >> 16), spare = e.y & 31;
  const bool two = (xa & 31) > spare;  // the window reaches into the next word
  const int q1 = (D.o1 >> 1) + (int)(short)(e.x & 0xffff), q2 = (D.o2 >> 1) + (e.x >> 16);
  const int half = (D.axis == 0 ? M.dim_vox[1] : M.dim_vox[0]) >> 1;  // row groups along o1
  const int rw = D.axis == 0 ? M.rw : (D.axis == 1 ? M.rw_y : M.rw_z);
  const int w = xa >> 5;
  uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
  if (FAST) {
    const int at = (q2 * half + q1) * rw + w;
    const size_t quads = D.axis == 0 ? M.quads : (D.axis == 1 ? M.quads_y : M.quads_z);
    if (!check_index(at >= 0 && (size_t)at + two < quads, M.ctl)) return lo;
    lo = __ldg(view + at);
    if (two) hi = __ldg(view + at + 1);
  } else {
    const int half2 = (D.axis == 2 ? M.dim_vox[1] : M.dim_vox[2]) >> 1;
    if ((unsigned)q1 < (unsigned)half && (unsigned)q2 < (unsigned)half2) {
      const uint4* row = view + ((size_t)q2 * half + q1) * rw;
      if ((unsigned)w < (unsigned)rw) lo = __ldg(row + w);
      if (two && (unsigned)(w + 1) < (unsigned)rw) hi = __ldg(row + w + 1);
    }
  }
  return make_uint4(__funnelshift_r(lo.x, hi.x, xa) & m.x, __funnelshift_r(lo.y, hi.y, xa) & m.y,
                    __funnelshift_r(lo.z, hi.z, xa) & m.z, __funnelshift_r(lo.w, hi.w, xa) & m.w);
}

__device__ __forceinline__ int popc4(uint4 b) {
  return __popc(b.x) + __popc(b.y) + __popc(b.z) + __popc(b.w);
}

// Lanes that count one direction: kSide directions are counted side by side. With
// 4 / 8 / 16 lanes 53.2 / 52.9 / 56.9 us per pine frame, 1.39 / 1.34 / 1.48 ms on
// the 1 cm map.
constexpr int kDirLanes = 8;
constexpr int kSide = 32 / kDirLanes;

// Occupied tool voxels, saturated at `sat`, of up to kSide directions side by
// side: the lanes of group k (lanes kDirLanes k on) count the direction of table
// entry `d` (equal over the group; none unless `valid`), one entry per lane per
// step, and all get its count. A group that has reached `sat` stops loading.
// One entry per lane, not two: entries come nearest first and most directions
// are decided by the first few, so wider steps load words that nobody needs
// (61 -> 52 us per pine frame together with the corridor's).
template <bool FAST>
__device__ inline int tool_counts(const MapView& M, const ToolView& T, bool valid, int4 d, const Pt& P,
                                  int sat, int lane) {
  DirRows D = dir_rows(M, P, d);
  if (!valid) D.nt = 0;
  int total = 0, b = lane & (kDirLanes - 1), left = D.nt;
  while (__any_sync(0xffffffffu, left > 0)) {
    int c = 0;
    if (left > 0 && b < D.nt) {
      uint4 m;
      c = popc4(quad_bits<FAST>(M, T, D, D.view, D.t0 + b, &m));
    }
#pragma unroll
    for (int off = kDirLanes / 2; off; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    total += c;
    b += kDirLanes;
    left = total < sat ? left - kDirLanes : 0;
  }
  return min(total, sat);
}

// Occupied tool voxels of direction g at point P, saturated at `sat`; the
// whole warp on one direction.
template <bool FAST>
__device__ inline int tool_count(const MapView& M, const ToolView& T, int g, const Pt& P, int sat,
                                 int lane) {
  const DirRows D = dir_rows(M, P, __ldg(T.dtab + g));
  int total = 0;
  for (int b = 0; b < D.nt && total < sat; b += 32) {
    uint4 m;
    const int c = b + lane < D.nt ? popc4(quad_bits<FAST>(M, T, D, D.view, D.t0 + b + lane, &m)) : 0;
    total += __reduce_add_sync(0xffffffffu, c);
  }
  return min(total, sat);
}

// Corridor of the direction of table entry d: any occupied voxel (strict: or
// unknown) blocks. The whole warp, one entry per lane per step (most blocked
// corridors are so by their nearest entries). Strict corridors run along x, the
// known view's rows.
template <bool FAST, bool STRICT>
__device__ inline bool corridor_blocked(const MapView& M, const ToolView& T, int4 d, const Pt& P,
                                        int lane) {
  const DirRows D = dir_rows(M, P, d, STRICT);
  for (int b = lane; b - lane < D.nc; b += 32) {
    bool h = false;
    if (b < D.nc) {
      uint4 m;
      const uint4 o = quad_bits<FAST>(M, T, D, D.view, D.c0 + b, &m);
      h = (o.x | o.y | o.z | o.w) != 0u;
      if (STRICT) {
        const uint4 n = quad_bits<FAST>(M, T, D, M.known, D.c0 + b, &m);
        h = h || ((n.x ^ m.x) | (n.y ^ m.y) | (n.z ^ m.z) | (n.w ^ m.w)) != 0u;
      }
    }
    if (__any_sync(0xffffffffu, h)) return true;
  }
  return false;
}

// The three arm samples of direction g (one lane): clear iff none is
// occupied or unknown. All loads are issued together (no short circuit), so
// the screen costs two dependent round trips, not up to nine. The two views
// share their layout, so one index serves both.
template <bool FAST>
__device__ inline bool arm_clear(const MapView& M, const ToolView& T, int g, const Pt& P) {
  uint32_t clear = 1u;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const short4 a = __ldg(T.arm + 3 * g + s);
    const int x = P.px + a.x, y = P.py + a.y, z = P.pz + a.z;
    uint32_t oc = 0u, kn = 0u;
    if (FAST || ((unsigned)x < (unsigned)M.dim_vox[0] && (unsigned)y < (unsigned)M.dim_vox[1] &&
                 (unsigned)z < (unsigned)M.dim_vox[2])) {
      const size_t at = FAST ? (size_t)(((z >> 1) * (M.dim_vox[1] >> 1) + (y >> 1)) * M.rw + (x >> 5))
                             : ((size_t)(z >> 1) * (M.dim_vox[1] >> 1) + (y >> 1)) * M.rw + (x >> 5);
      if (check_index(at < M.quads, M.ctl)) {
        const size_t word = 4 * at + parity(y, z);
        oc = __ldg(reinterpret_cast<const uint32_t*>(M.occ) + word);
        kn = __ldg(reinterpret_cast<const uint32_t*>(M.known) + word);
      }
    }
    clear &= (kn & ~oc) >> (x & 31);
  }
  return clear & 1u;
}

// Whether direction g (table entry d; one lane) is open at its start: its arm
// samples are clear and, in the strict form, its nearest corridor entry holds no
// unknown voxel. Beyond the cleared band most of a map's space is unknown, so that
// entry blocks most strict corridors, 32 directions at a time and before anything
// is counted. Left to the corridor walk, a warp step for each direction after its
// tool count, strict scoring took 213 us per pine frame (12k points, 128
// directions) and 2.71 ms for the 1 cm map with 512; with it and the order of
// best_direction 67 us and 0.35 ms.
template <bool FAST, bool STRICT>
__device__ inline bool start_open(const MapView& M, const ToolView& T, int g, int4 d, const Pt& P) {
  if (!arm_clear<FAST>(M, T, g, P)) return false;
  if (!STRICT || d.w == 0) return true;
  const DirRows D = dir_rows(M, P, d, true);
  uint4 m;
  const uint4 n = quad_bits<FAST>(M, T, D, M.known, D.c0, &m);
  return ((n.x ^ m.x) | (n.y ^ m.y) | (n.z ^ m.z) | (n.w ^ m.w)) == 0u;
}

__device__ inline bool candidate(const ToolView& T, int g, float n0, float n1, float n2) {
  if (g >= T.G) return false;
  const float u0 = __ldg(T.dirs + 3 * g), u1 = __ldg(T.dirs + 3 * g + 1),
              u2 = __ldg(T.dirs + 3 * g + 2);
  const float nu = __fadd_rn(__fadd_rn(__fmul_rn(n0, u0), __fmul_rn(n1, u1)), __fmul_rn(n2, u2));
  return nu > T.cos_max;
}

// The normal filter of Sec. 3.4 as a candidate test.
struct NormalFilter {
  float n0, n1, n2;
  __device__ bool operator()(const ToolView& T, int g) const { return candidate(T, g, n0, n1, n2); }
};

// The same with the masks of the first 1,024 directions kept, 32 per lane.
struct KeptFilter {
  NormalFilter F;
  unsigned kept;  // lane k: the candidates among directions 32 k .. 32 k + 31
  __device__ bool operator()(const ToolView& T, int g) const {
    const int group = g >> 5;  // one group for the whole warp
    if (group >= 32) return F(T, g);
    return (__shfl_sync(0xffffffffu, kept, group) >> (g & 31)) & 1u;
  }
};

struct NoGate {
  __device__ bool operator()() const { return true; }
};

__device__ __forceinline__ int4 shfl4(int4 v, int from) {
  return make_int4(__shfl_sync(0xffffffffu, v.x, from), __shfl_sync(0xffffffffu, v.y, from),
                   __shfl_sync(0xffffffffu, v.z, from), __shfl_sync(0xffffffffu, v.w, from));
}

// The candidate loop of one point: lowest-index minimum of the direction
// scores, with exact early exits; `cand(T, g)` says whether direction g is a
// candidate of the point. Returns (best score, best index), (n_c + 1, first
// candidate) if every candidate is blocked, (n_c + 2, -1) without candidates.
// `gate()` is asked once, after the first screen (so that a load it waits for
// overlaps the screen's): if it says no, (-1, -1) is returned.
//
// The screen (start_open) takes 32 directions at a time. The open ones are then
// counted kSide at a time, all against the score to beat before them, and
// decided in index order: a count that reaches that score cannot beat any later
// one, so the result is the sequential one. A score of 0 ends the search.
//
// STRICT: until a direction is found, the corridor comes before the count. Most
// strict corridors are blocked, and a count is only needed of one that is not.
// A template parameter, not a branch on the tool: both forms in one search cost the
// usual one 2 to 3%.
template <bool FAST, bool STRICT, class Cand, class Gate = NoGate>
__device__ inline int2 best_direction(const MapView& M, const ToolView& T, const Pt& P,
                                      const Cand& cand_of, int lane, const Gate& gate = Gate()) {
  const int nc = T.n_c;
  int bscore = nc + 1, best = -1, first = -1;  // best: of the unblocked directions
  for (int gb = 0; gb < T.G; gb += 32) {
    // lane-parallel screen: candidates, and the start of each candidate
    const bool cand = cand_of(T, gb + lane);
    const unsigned mask = __ballot_sync(0xffffffffu, cand);
    if (first < 0 && mask) first = gb + __ffs(mask) - 1;
    const int4 dt = cand ? __ldg(T.dtab + gb + lane) : make_int4(0, 0, 0, 0);
    unsigned rest = __ballot_sync(0xffffffffu, cand && start_open<FAST, STRICT>(M, T, gb + lane, dt, P));
    if (gb == 0 && !gate()) return make_int2(-1, -1);
    while (rest) {
      int at, c = 0;
      unsigned todo;
      const bool one = STRICT && best < 0;
      if (one) {  // the next open direction, not counted yet
        at = __ffs(rest) - 1;
        rest &= rest - 1u;
        todo = 1u;
      } else {
        // the next kSide open directions, one per group of lanes
        unsigned mine = rest;
#pragma unroll
        for (int k = 1; k < kSide; ++k) {
          if (lane >= k * kDirLanes) mine &= mine - 1u;
          rest &= rest - 1u;
        }
        rest &= rest - 1u;
        at = mine ? __ffs(mine) - 1 : 0;
        c = tool_counts<FAST>(M, T, mine != 0u, shfl4(dt, at), P, min(bscore, nc), lane);
        todo = __ballot_sync(0xffffffffu, mine != 0u && (best < 0 || c < bscore) &&
                                              (lane & (kDirLanes - 1)) == 0);
      }
      while (todo) {
        const int from = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int k = __shfl_sync(0xffffffffu, at, from);
        int ck = __shfl_sync(0xffffffffu, c, from);
        if (best >= 0 && ck >= bscore) continue;  // beaten by one before it
        if (corridor_blocked<FAST, STRICT>(M, T, shfl4(dt, k), P, lane)) continue;
        if (one) ck = tool_count<FAST>(M, T, gb + k, P, nc, lane);
        bscore = ck;
        best = gb + k;
        if (bscore == 0) return make_int2(0, best);
      }
    }
  }
  if (best >= 0) return make_int2(bscore, best);
  return first >= 0 ? make_int2(nc + 1, first) : make_int2(nc + 2, -1);
}

// best_direction with a budget: at most `budget` directions are taken past
// the screen (tool count and corridor). If the search stops early,
// *next receives the first direction index not searched and the result is
// exact over the directions before it; *next = -1 when the search finished.
template <bool FAST, bool STRICT, class Cand>
__device__ inline int2 best_direction_budget(const MapView& M, const ToolView& T, const Pt& P,
                                             const Cand& cand_of, int lane, int budget,
                                             int* next) {
  const int nc = T.n_c;
  int bscore = nc + 2, best = -1, spent = 0;
  *next = -1;
  for (int gb = 0; gb < T.G && bscore != 0; gb += 32) {
    const bool cand = cand_of(T, gb + lane);
    unsigned mask = __ballot_sync(0xffffffffu, cand);
    const int4 dt = cand ? __ldg(T.dtab + gb + lane) : make_int4(0, 0, 0, 0);
    const unsigned open =
        __ballot_sync(0xffffffffu, cand && start_open<FAST, STRICT>(M, T, gb + lane, dt, P));
    while (mask) {
      const int bit = __ffs(mask) - 1;
      const int g = gb + bit;
      mask &= mask - 1u;
      if (!((open >> bit) & 1u)) {
        if (best < 0) {
          bscore = nc + 1;
          best = g;
        }
        continue;
      }
      if (spent == budget) {
        *next = g;
        return make_int2(bscore, best);
      }
      ++spent;
      if (bscore <= nc) {
        const int cnt = tool_count<FAST>(M, T, g, P, bscore, lane);
        if (cnt >= bscore) continue;
        if (corridor_blocked<FAST, STRICT>(M, T, __ldg(T.dtab + g), P, lane)) continue;
        bscore = cnt;
        best = g;
      } else {
        if (corridor_blocked<FAST, STRICT>(M, T, __ldg(T.dtab + g), P, lane)) {
          if (best < 0) {
            bscore = nc + 1;
            best = g;
          }
          continue;
        }
        bscore = tool_count<FAST>(M, T, g, P, nc, lane);
        best = g;
      }
      if (bscore == 0) break;
    }
  }
  return make_int2(bscore, best);
}

// A (score, direction) result packed so that the lowest-index minimum is the
// smallest word: score in the high half, direction (0xFFFF: none) below.
__device__ inline uint32_t pack_result(int2 r) {
  return ((uint32_t)r.x << 16) | (r.y < 0 ? 0xFFFFu : (uint32_t)r.y);
}

}  // namespace af
