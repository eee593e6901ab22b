// af_noalloc.cu -- af_integrate_scan_noalloc: scan integration for callers
// that cannot allocate device memory.
//
// Some callers may not call cudaMalloc at all: a real-time loop whose memory
// is budgeted once at start-up, a host framework that owns every device
// buffer through its own arena, or code that must not enter the CUDA
// allocator while other work is in flight. af_create allocates the hashed
// map, so it is out of reach for them. This entry point integrates one scan
// into a dense voxel box that the caller owns and passes in; the only other
// memory it needs -- the per-return scratch that the allocating path keeps in
// its context -- lives in the file-scope device array below. The library
// itself allocates nothing here: no cudaMalloc, no cudaFree, no allocating
// library routine.
//
// The scratch array is AF_NOALLOC_MAX_RETURNS float4 (1 MiB). Every GPU that
// loads the library holds it until the process exits. All calls share it and
// it keeps the last call's contents; each call writes every element it reads
// before reading it, so nothing in it has to start at zero. Calls that
// overlap on the GPU (on different streams, or from several threads) race on
// the array: serialise them.
#include <af.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <mutex>

#include "af_cube.cuh"
#include "af_internal.cuh"

namespace af {
void set_global_error(const char* msg);  // af_last_error(NULL) reports it

namespace {

static __device__ __align__(256) float4 g_scan_scratch[AF_NOALLOC_MAX_RETURNS];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
float4* g_scratch_dev[kMaxDevices] = {nullptr};  // device address of the array, per device
af_status nfail(af_status s, const char* fmt, ...) {
  char buf[256];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  set_global_error(buf);
  return s;
}

// Device address of the scratch array on the current device; looked up once
// per device (the host-side name of the array is not a device address).
af_status scratch_address(float4** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return nfail(AF_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return nfail(AF_ERR_CUDA, "device index %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_dev[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_scan_scratch);
    if (e != cudaSuccess || !p)
      return nfail(AF_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    g_scratch_dev[dev] = static_cast<float4*>(p);
  }
  *out = g_scratch_dev[dev];
  return AF_OK;
}

struct Box {
  int lo[3];       // domain-relative voxel index of the box corner
  int dim[3];
  unsigned long long* vox;
  uint8_t* flags;
};

__device__ inline bool box_index(const Box& B, int x, int y, int z, size_t* at) {
  x -= B.lo[0];
  y -= B.lo[1];
  z -= B.lo[2];
  if ((unsigned)x >= (unsigned)B.dim[0] || (unsigned)y >= (unsigned)B.dim[1] ||
      (unsigned)z >= (unsigned)B.dim[2])
    return false;
  *at = ((size_t)z * B.dim[1] + y) * B.dim[0] + x;
  return true;
}

// Box offset of the coordinate with domain-relative index j on axis ax (the
// three axes' offsets add up to the voxel's element), or -1 outside the box.
__device__ inline long long box_offset(const Box& B, int ax, int j) {
  j -= B.lo[ax];
  if ((unsigned)j >= (unsigned)B.dim[ax]) return -1;
  return ax == 0 ? (long long)j
                 : (ax == 1 ? (long long)j * B.dim[0] : (long long)j * ((long long)B.dim[0] * B.dim[1]));
}

// One CTA per T returns, one thread per cube offset: the returns are
// transformed and their per-axis terms and box offsets computed once into
// shared memory, then each thread walks the returns for its offset, the same
// arithmetic as the hashed path (af_cube.cuh), one 64-bit atomic add per pair;
// the cleared-band marks follow. The world positions go to `scratch` for
// k_box_finalize. Issue-bound like k_integrate: 26.3 us per pine frame; with one
// thread per (return, offset) that did all of a pair's work, 64-bit divisions
// included, for itself, 73 us and a launch for the transform.
template <int W, int T>
__global__ void __launch_bounds__(CubeShape<W>::NT) k_box_integrate(MapView M,
                                                                    const float* __restrict__ xyz,
                                                                    uint32_t n, Pose P,
                                                                    float4* __restrict__ scratch,
                                                                    Box B) {
  using S = CubeShape<W>;
  __shared__ float4 s_p[T], s_pr[T];
  __shared__ float4 s_term[T][3][W];
  __shared__ long long s_off[T][3][W];
  const int tid = threadIdx.x;
  const uint32_t r0 = blockIdx.x * T;
  const float q[3] = {P.r[0][3], P.r[1][3], P.r[2][3]};
  if (tid < T) {
    const uint32_t k = r0 + tid;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < n) {
      float w[3], range;
      int rel[3];
      const bool valid = prepare_return(M, P, xyz[3 * k], xyz[3 * k + 1], xyz[3 * k + 2], w, &range, rel);
      p = valid ? make_float4(w[0], w[1], w[2], 1.f) : p;
      scratch[k] = p;
    }
    s_p[tid] = p;
    s_pr[tid] = return_record(p, q[0], q[1], q[2]);
  }
  __syncthreads();
  for (int e = tid; e < T * 3 * W; e += S::NT) {
    const int t = e / (3 * W), ax = (e / W) % 3, k = e % W;
    const float4 p = s_p[t];
    if (p.w == 0.f) continue;
    const float pa = ax == 0 ? p.x : (ax == 1 ? p.y : p.z);
    int i;
    voxel_index(pa, M, &i);  // accepted by prepare_return
    s_term[t][ax][k] = axis_terms(M, pa, q[ax], i + k - S::MR);
    s_off[t][ax][k] = box_offset(B, ax, i - M.dom_vox[ax] + k - S::MR);
  }
  __syncthreads();
  int kx[S::OPT], ky[S::OPT], kz[S::OPT];  // ox fastest: neighbouring threads, neighbouring words
#pragma unroll
  for (int s = 0; s < S::OPT; ++s) {
    const int o = tid + s * S::NT;
    kx[s] = o % W;
    ky[s] = (o / W) % W;
    kz[s] = o / (W * W);
  }
  for (int t = 0; t < T; ++t) {
    const float4 pr = s_pr[t];
    if (pr.w == 0.f) continue;  // uniform across the block
#pragma unroll
    for (int s = 0; s < S::OPT; ++s) {
      if (tid + s * S::NT >= S::C) break;
      long long dq;
      if (!pair_contribution(M, s_term[t][0][kx[s]], s_term[t][1][ky[s]], s_term[t][2][kz[s]], pr, &dq))
        continue;
      const long long ox = s_off[t][0][kx[s]], oy = s_off[t][1][ky[s]], oz = s_off[t][2][kz[s]];
      if ((ox | oy | oz) >= 0) atomicAdd(B.vox + (ox + oy + oz), make_word(dq, 1ull));
    }
  }
  for (int e = tid; e < T * M.ns; e += S::NT) {
    const int t = e / M.ns, s = e % M.ns + 1;
    if (s_p[t].w == 0.f) continue;
    const float p[3] = {s_p[t].x, s_p[t].y, s_p[t].z};
    int sv[3];
    size_t at;
    if (band_sample(M, p, q, s_pr[t].x, s, sv) && box_index(B, sv[0], sv[1], sv[2], &at))
      B.flags[at] |= 1u;  // every writer sets bit 0
  }
}

// Weight cap and occupied / known flags of box voxel `at`. Idempotent (a
// capped weight is not capped again), so threads that reach the same voxel
// through different returns write the same word and flags; a voxel that another
// thread has done is read but not written.
__device__ inline void finalize_voxel(const MapView& M, const Box& B, size_t at) {
  unsigned long long word = B.vox[at];
  unsigned long long w = word & kWMask;
  long long S = word_S(word);
  if (w > M.w_cap) {
    S = capped_S(S, M.w_cap, (long long)w);
    w = M.w_cap;
    B.vox[at] = make_word(S, w);
  }
  const unsigned was = B.flags[at], cl = was & 1u;
  const unsigned occ = (w >= 1 && S < (long long)M.rcq * (long long)w) ? 1u : 0u;
  const unsigned kn = (w >= 1 || cl) ? 1u : 0u;
  const unsigned now = cl | (occ << 1) | (kn << 2);
  if (now != was) B.flags[at] = (uint8_t)now;
}

// Weight cap and flags of every voxel this scan touched -- the cube voxels
// and cleared-band samples of its accepted returns, enumerated as in
// k_box_integrate -- after all of the scan's additions (a launch of its own).
// Voxels the scan does not touch keep their words and flags. A voxel is reached
// through many returns: bound by the L2 reads of its word and flags (29 us per
// pine frame; one thread per (return, offset) that found its voxel by itself and
// always wrote the flags took 117 us).
template <int W, int T>
__global__ void __launch_bounds__(CubeShape<W>::NT) k_box_finalize(MapView M,
                                                                   const float4* __restrict__ scratch,
                                                                   uint32_t n, float q0, float q1,
                                                                   float q2, Box B) {
  using S = CubeShape<W>;
  __shared__ float4 s_p[T];
  __shared__ long long s_off[T][3][W];
  const int tid = threadIdx.x;
  const uint32_t r0 = blockIdx.x * T;
  for (int e = tid; e < T * 3 * W; e += S::NT) {
    const int t = e / (3 * W), ax = (e / W) % 3, k = e % W;
    const float4 p = r0 + t < n ? scratch[r0 + t] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (ax == 0 && k == 0) s_p[t] = p;
    if (p.w == 0.f) continue;
    int i;
    voxel_index(ax == 0 ? p.x : (ax == 1 ? p.y : p.z), M, &i);
    s_off[t][ax][k] = box_offset(B, ax, i - M.dom_vox[ax] + k - S::MR);
  }
  __syncthreads();
  for (int t = 0; t < T; ++t) {
    if (s_p[t].w == 0.f) continue;
#pragma unroll
    for (int s = 0; s < S::OPT; ++s) {
      const int o = tid + s * S::NT;
      if (o >= S::C) break;
      const long long ox = s_off[t][0][o % W], oy = s_off[t][1][(o / W) % W], oz = s_off[t][2][o / (W * W)];
      if ((ox | oy | oz) >= 0) finalize_voxel(M, B, (size_t)(ox + oy + oz));
    }
  }
  const float q[3] = {q0, q1, q2};
  for (int e = tid; e < T * M.ns; e += S::NT) {
    const int t = e / M.ns, s = e % M.ns + 1;
    if (s_p[t].w == 0.f) continue;
    const float p[3] = {s_p[t].x, s_p[t].y, s_p[t].z};
    int sv[3];
    size_t at;
    if (band_sample(M, p, q, return_record(s_p[t], q0, q1, q2).x, s, sv) &&
        box_index(B, sv[0], sv[1], sv[2], &at))
      finalize_voxel(M, B, at);
  }
}

template <int W, int T>
void launch_box_tile(const MapView& M, const float* xyz, uint32_t n, const Pose& P, float4* scratch,
                     const Box& B, cudaStream_t s) {
  const unsigned grid = (n + T - 1) / T;
  k_box_integrate<W, T><<<grid, CubeShape<W>::NT, 0, s>>>(M, xyz, n, P, scratch, B);
  k_box_finalize<W, T><<<grid, CubeShape<W>::NT, 0, s>>>(M, scratch, n, P.r[0][3], P.r[1][3], P.r[2][3], B);
}

template <int W>
void launch_box(const MapView& M, const float* xyz, uint32_t n, const Pose& P, float4* scratch,
                const Box& B, cudaStream_t s) {
  const int T = tile_of<W>(n, kSetupBox);
  if constexpr (W > 5) {
    if (T == 16) return launch_box_tile<W, 16>(M, xyz, n, P, scratch, B, s);
    if (T == 12) return launch_box_tile<W, 12>(M, xyz, n, P, scratch, B, s);
  }
  if constexpr (W > 3) {
    if (T == 8) return launch_box_tile<W, 8>(M, xyz, n, P, scratch, B, s);
  }
  launch_box_tile<W, 4>(M, xyz, n, P, scratch, B, s);
}

bool finite_f(float x) { return std::isfinite(x); }

}  // namespace
}  // namespace af

extern "C" af_status af_integrate_scan_noalloc(const af_config* cfg, const float* d_xyz,
                                               uint32_t n, const float pose[16],
                                               const int32_t box_min[3], const uint32_t box_dim[3],
                                               uint64_t* d_vox, uint8_t* d_flags, void* stream) {
  using namespace af;
  if (!cfg || !pose || !box_min || !box_dim || !d_vox || !d_flags || (n > 0 && !d_xyz))
    return nfail(AF_ERR_INVALID_ARG, "af_integrate_scan_noalloc: NULL argument");
  if (n > AF_NOALLOC_MAX_RETURNS)
    return nfail(AF_ERR_CAPACITY,
                 "af_integrate_scan_noalloc: n = %u returns exceeds the fixed scratch of %d "
                 "returns; split the scan",
                 n, AF_NOALLOC_MAX_RETURNS);
  const float f[8] = {cfg->voxel_size, cfg->truncation, cfg->r_c,      cfg->cone_cos,
                      cfg->range_min,  cfg->range_max,  cfg->clear_lo, cfg->clear_hi};
  for (float x : f)
    if (!finite_f(x)) return nfail(AF_ERR_INVALID_ARG, "af_integrate_scan_noalloc: non-finite parameter");
  if (!(cfg->voxel_size > 0.f) || !(cfg->truncation > 0.f && cfg->truncation <= 1.f) ||
      !(cfg->r_c > 0.f && cfg->r_c <= 1.f) || cfg->cube_radius < 1 || cfg->cube_radius > 8 ||
      cfg->clear_samples < 0 || cfg->clear_samples > 64 || cfg->block_edge != 8 ||
      cfg->w_cap < 1 || (uint64_t)AF_NOALLOC_MAX_RETURNS + cfg->w_cap >= (1ull << kWBits) ||
      !(cfg->range_max > cfg->range_min) || !(cfg->clear_hi >= cfg->clear_lo) ||
      (cfg->clamp_signed != 0 && cfg->clamp_signed != 1))
    return nfail(AF_ERR_INVALID_ARG, "af_integrate_scan_noalloc: parameter out of range");
  uint64_t count = 1;
  for (int k = 0; k < 3; ++k) {
    if (cfg->domain_bricks[k] < 1 || cfg->domain_bricks[k] >= (1u << 21) ||
        std::abs((long long)cfg->domain_min[k]) > (1 << 25) || box_dim[k] < 1 ||
        box_dim[k] >= (1u << 24) || std::abs((long long)box_min[k]) > (1 << 28))
      return nfail(AF_ERR_INVALID_ARG, "af_integrate_scan_noalloc: domain or box out of range");
    // each factor is below 2^24, so the running product (at most 2^40 before
    // this step) cannot wrap before the check
    count *= box_dim[k];
    if (count > AF_NOALLOC_MAX_BOX_VOXELS)
      return nfail(AF_ERR_INVALID_ARG,
                   "af_integrate_scan_noalloc: the box holds more than 2^40 voxels");
  }
  for (int k = 0; k < 12; ++k)
    if (!finite_f(pose[k])) return nfail(AF_ERR_INVALID_ARG, "af_integrate_scan_noalloc: non-finite pose");

  float4* scratch = nullptr;
  af_status st = scratch_address(&scratch);
  if (st != AF_OK) return st;

  MapView M{};
  M.v = cfg->voxel_size;
  M.inv_v = 1.0f / cfg->voxel_size;
  M.tau = cfg->truncation;
  M.r_c = cfg->r_c;
  M.cone_cos = cfg->cone_cos;
  M.range_min = cfg->range_min;
  M.range_max = cfg->range_max;
  M.clear_lo = cfg->clear_lo;
  M.clear_hi = cfg->clear_hi;
  M.m = cfg->cube_radius;
  M.ns = cfg->clear_samples;
  M.w_min = cfg->w_min;
  M.w_cap = cfg->w_cap;
  M.rcq = (uint64_t)rintf(cfg->r_c * kScale);
  M.clamp_signed = cfg->clamp_signed;
  M.dlo = cfg->clamp_signed ? -cfg->truncation : 0.f;
  for (int k = 0; k < 3; ++k) {
    M.dom_vox[k] = cfg->domain_min[k] * 8;
    M.dim_vox[k] = (int)cfg->domain_bricks[k] * 8;
  }
  Box B;
  for (int k = 0; k < 3; ++k) {
    B.lo[k] = box_min[k] - M.dom_vox[k];
    B.dim[k] = (int)box_dim[k];
  }
  B.vox = reinterpret_cast<unsigned long long*>(d_vox);
  B.flags = d_flags;
  Pose P;
  for (int r = 0; r < 3; ++r)
    for (int c = 0; c < 4; ++c) P.r[r][c] = pose[4 * r + c];

  cudaStream_t s = (cudaStream_t)stream;
  if (n > 0) {
    switch (2 * M.m + 1) {
#define AF_CASE(W) \
  case W: launch_box<W>(M, d_xyz, n, P, scratch, B, s); break;
      AF_CASE(3) AF_CASE(5) AF_CASE(7) AF_CASE(9) AF_CASE(11) AF_CASE(13) AF_CASE(15) AF_CASE(17)
#undef AF_CASE
    }
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return nfail(AF_ERR_CUDA, "af_integrate_scan_noalloc: launch failed: %s",
                                     cudaGetErrorString(e));
  return AF_OK;
}

