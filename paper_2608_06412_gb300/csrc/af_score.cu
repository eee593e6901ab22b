// af_score.cu -- accessibility scoring on sm_103a (Sec. 3.4, 3.5 of the paper).
//
// One warp per surface point.
// The lanes first evaluate the normal filter for
// 32 directions at a time (ballot -> candidate mask), then the start of each
// candidate (the three arm samples, single-bit lookups: occupied or unknown
// blocks; with strict corridors their nearest entry too). The open candidates are
// taken four at a time (kSide) in index order:
//   * tool kernel: 8 lanes per direction fetch the kernel's entries (the same
//     32 voxels of four rows in one or two 16-byte loads), AND with the masks
//     and __popc; the count saturates at the score to beat, so it stops as
//     soon as the direction can no longer improve the point;
//   * corridor: the whole warp, one entry per lane per step, any set bit
//     blocks (__any_sync early exit).
// The best direction is the lowest-index minimum; a score of 0 ends the
// point. Every early exit returns exactly what a full evaluation of every
// candidate would (the score to beat only shrinks; ties keep the lower
// index).
//
// Work sharing (ScoreSplit): a point whose search takes more than `budget`
// directions past the screen stops there and hands the rest of its
// directions to k_score_split, where one warp takes each (point, direction)
// item, prunes it against the point's packed best so far (read at the start
// of the item; the best only ever decreases) and folds its exact score in
// with atomicMin. The packed lowest-index minimum is the result of the full
// search whatever the order the items run in; k_score_finish writes it out.
// The split bounds the span of the launch by the heaviest direction instead
// of the heaviest point.
//
// The device functions live in af_score.cuh.
#include <algorithm>

#include "af_score.cuh"

namespace af {

// Scores point pi with the whole warp (all 32 lanes call this together).
template <bool SPLIT, bool STRICT>
__device__ void score_point(const MapView& M, const ToolView& T, const float* __restrict__ pts,
                            const float* __restrict__ nrm, uint32_t pi,
                            uint8_t* __restrict__ label, int16_t* __restrict__ best_out,
                            int lane, const ScoreSplit& S) {
  const float s0 = pts[3 * pi], s1 = pts[3 * pi + 1], s2 = pts[3 * pi + 2];
  const float n0 = nrm[3 * pi], n1 = nrm[3 * pi + 1], n2 = nrm[3 * pi + 2];

  // The point's voxel and its weight (confidence gate, Sec. 3.5). Three
  // dependent loads lead to the weight (point, hash slot, voxel word): the
  // slot's is in flight while the candidates are found, the word's while the
  // first directions are screened.
  int i0 = 0, i1 = 0, i2 = 0;
  const bool ok =
      voxel_index(s0, M, &i0) && voxel_index(s1, M, &i1) && voxel_index(s2, M, &i2);
  Pt P;
  P.px = i0 - M.dom_vox[0];
  P.py = i1 - M.dom_vox[1];
  P.pz = i2 - M.dom_vox[2];
  const bool in = ok && (unsigned)P.px < (unsigned)M.dim_vox[0] &&
                  (unsigned)P.py < (unsigned)M.dim_vox[1] && (unsigned)P.pz < (unsigned)M.dim_vox[2];
  const uint64_t key = in ? pack_brick(P.px >> 3, P.py >> 3, P.pz >> 3) : kEmptyKey;
  unsigned long long found = kEmptyKey;
  uint32_t blk = kNoBlock, stamp;
  if (in) load_slot(M, hash_slot(key, M.hmask), &found, &blk, &stamp);

  // nominal tests: every candidate direction of this point
  int ncand = 0;
  KeptFilter F{{n0, n1, n2}, 0u};
  for (int gb = 0; gb < T.G; gb += 32) {
    const unsigned m = __ballot_sync(0xffffffffu, candidate(T, gb + lane, n0, n1, n2));
    ncand += __popc(m);
    if (lane == gb >> 5) F.kept = m;
  }

  if (found != key) blk = found == kEmptyKey ? kNoBlock : lookup_brick(M, key);  // the same in all lanes
  unsigned long long word = 0;
  if (in && blk < M.pool_blocks)
    word = __ldcg(M.vox + (size_t)blk * kBrickVox + ((P.px & 7) | ((P.py & 7) << 3) | ((P.pz & 7) << 6)));
  const auto confident = [&] { return (uint32_t)(word & kWMask) >= M.w_min; };

  const bool fast = reach_inside(M, T, P);
  int2 res;
  int next = -1;
  if (!SPLIT) {
    res = fast ? best_direction<true, STRICT>(M, T, P, F, lane, confident)
               : best_direction<false, STRICT>(M, T, P, F, lane, confident);
  } else {
    res = make_int2(-1, -1);
    if (confident())
      res = fast ? best_direction_budget<true, STRICT>(M, T, P, F, lane, S.budget, &next)
                 : best_direction_budget<false, STRICT>(M, T, P, F, lane, S.budget, &next);
  }
  if (res.x < 0) {  // not confident
    if (lane == 0) {
      label[pi] = 0;
      best_out[pi] = -1;
    }
    return;
  }

  if (lane == 0) {
    if (next < 0) {
      label[pi] = (res.y >= 0 && res.x < T.n_c) ? 1 : 2;
      best_out[pi] = (int16_t)res.y;
    } else {  // hand the directions from `next` on to k_score_split
      const uint32_t o = atomicAdd(S.count, 1u);
      S.over[o] = make_int2((int)pi, next);
      S.res[o] = pack_result(res);
    }
    atomicAdd(&M.ctl->points_scored, 1ull);
    atomicAdd(&M.ctl->tests, (unsigned long long)ncand);
  }
}

// Threads per SM the scorers are built for: 40 warps at 48 registers. Fewer warps
// hide less latency, more spill: 32 / 40 / 48 / 64 warps take 55.9 / 52.9 / 54.7 /
// 61.8 us per pine frame, 1.50 / 1.34 / 1.38 / 1.48 ms on the 1 cm map.
constexpr int kScoreThreads = 1280;

template <int WARPS, bool SPLIT, bool STRICT>
__global__ void __launch_bounds__(WARPS * 32, kScoreThreads / (WARPS * 32))
    k_score(MapView M, ToolView T, const float* __restrict__ pts, const float* __restrict__ nrm,
            uint32_t m, uint8_t* __restrict__ label, int16_t* __restrict__ best_out,
            ScoreSplit S) {
  const uint32_t pi = blockIdx.x * WARPS + (threadIdx.x >> 5);
  if (pi >= m) return;  // whole warp
  score_point<SPLIT, STRICT>(M, T, pts, nrm, pi, label, best_out, threadIdx.x & 31, S);
}

// One (point, direction) item of a handed-off search; the whole warp.
template <bool FAST, bool STRICT>
__device__ void split_item(const MapView& M, const ToolView& T, const Pt& P, int g, uint32_t* res,
                           int lane) {
  const int nc = T.n_c;
  const uint32_t cur = __ldcg(res);
  const int bs = (int)(cur >> 16), bg = (int)(cur & 0xFFFFu);  // bg 0xFFFF: none yet
  const int4 dt = __ldg(T.dtab + g);
  bool open = false;
  if (lane == 0) open = start_open<FAST, STRICT>(M, T, g, dt, P);
  open = __shfl_sync(0xffffffffu, open, 0);
  uint32_t mine;
  if (!open) {
    if (bs <= nc) return;  // blocked (n_c + 1) cannot beat an unblocked best
    mine = pack_result(make_int2(nc + 1, g));
  } else {
    // counts below `sat` may improve the best; `exact` counts up to n_c
    const bool exact = bs > nc || (g < bg && bs == nc);
    const int sat = exact ? nc : (g < bg ? bs + 1 : bs);
    if (!exact && sat == 0) return;
    const int c = tool_count<FAST>(M, T, g, P, sat, lane);
    if (!exact && c >= sat) return;
    mine = corridor_blocked<FAST, STRICT>(M, T, dt, P, lane) ? pack_result(make_int2(nc + 1, g))
                                                             : pack_result(make_int2(min(c, nc), g));
  }
  if (lane == 0 && mine < cur) atomicMin(res, mine);
}

template <bool STRICT>
__global__ void __launch_bounds__(128, kScoreThreads / 128)
    k_score_split(MapView M, ToolView T, const float* __restrict__ pts,
                  const float* __restrict__ nrm, ScoreSplit S) {
  const int lane = threadIdx.x & 31;
  const uint64_t items = (uint64_t)__ldcg(S.count) * (uint64_t)T.G;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t it = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nw) {
    const uint32_t o = (uint32_t)(it / (uint64_t)T.G);
    const int g = (int)(it - (uint64_t)o * T.G);
    const int2 ov = __ldcg(S.over + o);
    if (g < ov.y) continue;
    const uint32_t pi = (uint32_t)ov.x;
    if (!candidate(T, g, nrm[3 * pi], nrm[3 * pi + 1], nrm[3 * pi + 2])) continue;
    // the point passed the gate in k_score, so its voxel is inside the box
    int i0, i1, i2;
    voxel_index(pts[3 * pi], M, &i0);
    voxel_index(pts[3 * pi + 1], M, &i1);
    voxel_index(pts[3 * pi + 2], M, &i2);
    Pt P;
    P.px = i0 - M.dom_vox[0];
    P.py = i1 - M.dom_vox[1];
    P.pz = i2 - M.dom_vox[2];
    const bool fast = reach_inside(M, T, P);
    if (fast)
      split_item<true, STRICT>(M, T, P, g, S.res + o, lane);
    else
      split_item<false, STRICT>(M, T, P, g, S.res + o, lane);
  }
}

__global__ void __launch_bounds__(256) k_score_finish(ScoreSplit S, int n_c,
                                                      uint8_t* __restrict__ label,
                                                      int16_t* __restrict__ best_out) {
  const uint32_t n = __ldcg(S.count);
  for (uint32_t o = blockIdx.x * blockDim.x + threadIdx.x; o < n; o += gridDim.x * blockDim.x) {
    const uint32_t r = S.res[o];
    const uint32_t pi = (uint32_t)S.over[o].x;
    const int sc = (int)(r >> 16), g = (int)(r & 0xFFFFu);
    best_out[pi] = g == 0xFFFF ? (int16_t)-1 : (int16_t)g;
    label[pi] = (g != 0xFFFF && sc < n_c) ? 1 : 2;
  }
}

template <bool STRICT>
static cudaError_t launch_score_form(const MapView& M, const ToolView& T, const float* d_pts,
                                     const float* d_nrm, uint32_t m, uint8_t* d_label,
                                     int16_t* d_best, const ScoreSplit& S, int num_sms,
                                     cudaStream_t stream) {
  constexpr int WARPS = 2;
  const unsigned grid = (m + WARPS - 1) / WARPS;
  if (S.budget < 0) {
    k_score<WARPS, false, STRICT><<<grid, WARPS * 32, 0, stream>>>(M, T, d_pts, d_nrm, m, d_label,
                                                                   d_best, S);
    return cudaGetLastError();
  }
  const cudaError_t e = cudaMemsetAsync(S.count, 0, sizeof(uint32_t), stream);
  if (e != cudaSuccess) return e;
  k_score<WARPS, true, STRICT><<<grid, WARPS * 32, 0, stream>>>(M, T, d_pts, d_nrm, m, d_label,
                                                                d_best, S);
  k_score_split<STRICT><<<num_sms * (kScoreThreads / 128), 128, 0, stream>>>(M, T, d_pts, d_nrm, S);
  k_score_finish<<<num_sms, 256, 0, stream>>>(S, T.n_c, d_label, d_best);
  return cudaGetLastError();
}

cudaError_t launch_score(const MapView& M, const ToolView& T, const float* d_pts,
                         const float* d_nrm, uint32_t m, uint8_t* d_label, int16_t* d_best,
                         const ScoreSplit& S, int num_sms, cudaStream_t stream) {
  if (m == 0) return cudaSuccess;
  return T.strict ? launch_score_form<true>(M, T, d_pts, d_nrm, m, d_label, d_best, S, num_sms, stream)
                  : launch_score_form<false>(M, T, d_pts, d_nrm, m, d_label, d_best, S, num_sms, stream);
}

// Batched ticks: every point of every map of the batch, one warp per point,
// persistent grid (see af_batch.cu).
template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32, kScoreThreads / (WARPS * 32))
    k_score_batch(const BatchHdr* __restrict__ B, const SceneDesc* __restrict__ D) {
  const uint32_t total = B->total_points;
  const int count = (int)B->count;
  const uint32_t nw = gridDim.x * WARPS;
  for (uint32_t pg = blockIdx.x * WARPS + (threadIdx.x >> 5); pg < total; pg += nw) {
    const int s = scene_of<2>(D, count, pg);
    const SceneDesc& d = D[s];
    const ScoreSplit S{nullptr, nullptr, nullptr, -1};
    if (d.T.strict)
      score_point<false, true>(d.M, d.T, d.pts, d.nrm, pg - d.pt_off, d.label, d.best,
                               threadIdx.x & 31, S);
    else
      score_point<false, false>(d.M, d.T, d.pts, d.nrm, pg - d.pt_off, d.label, d.best,
                                threadIdx.x & 31, S);
  }
}

template <int WARPS>
static cudaError_t launch_score_batch_w(const BatchHdr* B, const SceneDesc* D, int num_sms,
                                        cudaStream_t stream) {
  int per = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_score_batch<WARPS>, WARPS * 32, 0);
  k_score_batch<WARPS><<<num_sms * (per > 0 ? per : 1), WARPS * 32, 0, stream>>>(B, D);
  return cudaGetLastError();
}

cudaError_t launch_score_batch(const BatchHdr* B, const SceneDesc* D, int warps, int num_sms,
                               cudaStream_t stream) {
  switch (warps) {
    case 2: return launch_score_batch_w<2>(B, D, num_sms, stream);
    case 4: return launch_score_batch_w<4>(B, D, num_sms, stream);
    case 8: return launch_score_batch_w<8>(B, D, num_sms, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace af
