// Padded batches for dense-attention consumers (Section 4, Analyses: the
// images of a batch are padded to the longest merged sequence and the
// padding is masked out).  pad_kernel writes [batch, L, dim] from the packed
// rows plus a key mask and the batch's N_b statistics; unpad_kernel is the
// inverse.  Both are bandwidth-bound copies: a warp takes a run of rows of one
// image, contiguous on both sides, and copies it as one sequence of 16-byte
// vectors.  A warp per row left most lanes of short rows idle and paid a
// 64-bit division per row: both copies of 1000 images of up to 300 rows of 64
// bf16 took 103.6 us and take 29.0, of 256 images of up to 256 rows of 384 32.8
// and 31.3, of 64 images of up to 877 rows of 768 53.5 and 52.7.
#include "mpm.h"
#include "common.cuh"
#include "launch.h"

namespace mpm {
namespace {

constexpr int kThreads = 256;
constexpr int kVecs = 6;  // 16-byte vectors in flight per lane (4: 52.7 -> 53.2 us for 64 x 877 x 768, 12: 53.8)
__device__ __forceinline__ int64_t clamp_off(int64_t v, int64_t rows) { return v < 0 ? 0 : (v > rows ? rows : v); }

// A run of up to `per_warp` consecutive rows of one padded image: its source
// and destination are both contiguous.
struct Run {
  int image;
  int64_t first;   // first padded row of the run within its image
  int64_t packed;  // the image's first packed row
  int64_t length;  // the image's packed rows
  int rows, live;  // padded rows of the run, and those of them that hold tokens
};
__device__ __forceinline__ Run locate_run(int64_t run, int64_t per_image, int per_warp, int64_t max_len,
                                          const int64_t* __restrict__ offsets, int64_t rows) {
  Run r;
  // The short 32-bit division where it is enough.
  r.image = ((run | per_image) >> 32) == 0
                ? static_cast<int>(static_cast<uint32_t>(run) / static_cast<uint32_t>(per_image))
                : static_cast<int>(run / per_image);
  r.first = (run - r.image * per_image) * per_warp;
  r.packed = clamp_off(__ldg(offsets + r.image), rows);
  r.length = clamp_off(__ldg(offsets + r.image + 1), rows) - r.packed;
  r.rows = static_cast<int>(max_len - r.first < per_warp ? max_len - r.first : per_warp);
  const int64_t left = r.length - r.first;
  r.live = static_cast<int>(left < 0 ? 0 : left < r.rows ? left : r.rows);
  return r;
}

// dst[0 .. n) = src[0 .. n), by one warp.
__device__ __forceinline__ void copy_vectors(uint4* __restrict__ dst, const uint4* __restrict__ src, int n, int lane) {
  for (int v0 = lane; v0 < n; v0 += 32 * kVecs) {
    uint4 val[kVecs];
#pragma unroll
    for (int u = 0; u < kVecs; ++u)
      if (v0 + 32 * u < n) val[u] = __ldg(src + v0 + 32 * u);
#pragma unroll
    for (int u = 0; u < kVecs; ++u)
      if (v0 + 32 * u < n) dst[v0 + 32 * u] = val[u];
  }
}

// out[b, t] = tokens[off_b + t] for t < min(N_b, L), zero rows after;
// mask[b, t] = 1 for the copied rows.  Block 0 also reduces N_b to
// (min, max, total) into stats.  An image longer than L is cut and reported.
__global__ void __launch_bounds__(kThreads) pad_kernel(const uint8_t* __restrict__ tokens,
                                                       const int64_t* __restrict__ offsets, int batch,
                                                       int64_t rows, int64_t max_len, int nvec,
                                                       int per_warp, uint8_t* __restrict__ out, uint8_t* __restrict__ mask,
                                                       int64_t* __restrict__ stats, int32_t* status) {
  wait_for_previous_grid();
  if (blockIdx.x == 0 && stats != nullptr) {
    __shared__ int64_t sh_min[kThreads / 32], sh_max[kThreads / 32], sh_sum[kThreads / 32];
    int64_t mn = INT64_MAX, mx = 0, sm = 0;
    for (int b = threadIdx.x; b < batch; b += kThreads) {
      const int64_t n = clamp_off(offsets[b + 1], rows) - clamp_off(offsets[b], rows);
      const int64_t nn = n > 0 ? n : 0;
      mn = nn < mn ? nn : mn;
      mx = nn > mx ? nn : mx;
      sm += nn;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const int64_t a = __shfl_xor_sync(0xFFFFFFFFu, mn, d), c = __shfl_xor_sync(0xFFFFFFFFu, mx, d);
      mn = a < mn ? a : mn;
      mx = c > mx ? c : mx;
      sm += __shfl_xor_sync(0xFFFFFFFFu, sm, d);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      sh_min[w] = mn;
      sh_max[w] = mx;
      sh_sum[w] = sm;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int i = 1; i < kThreads / 32; ++i) {
        mn = sh_min[i] < mn ? sh_min[i] : mn;
        mx = sh_max[i] > mx ? sh_max[i] : mx;
        sm += sh_sum[i];
      }
      stats[0] = batch > 0 ? mn : 0;
      stats[1] = mx;
      stats[2] = sm;
    }
  }
  const int lane = threadIdx.x & 31;
  const int64_t warp = (static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * kThreads) >> 5;
  const int64_t per_image = (max_len + per_warp - 1) / per_warp, runs = batch * per_image;
  for (int64_t run = warp; run < runs; run += nwarps) {
    const Run r = locate_run(run, per_image, per_warp, max_len, offsets, rows);
    if (r.first == 0 && lane == 0 && r.length > max_len) report(status, MPM_ERR_DEVICE_CHECK, r.image);
    const int64_t q0 = r.image * max_len + r.first;
    if (mask != nullptr && lane < r.rows) mask[q0 + lane] = lane < r.live ? 1 : 0;
    const uint4* src = reinterpret_cast<const uint4*>(tokens) + (r.packed + r.first) * nvec;
    uint4* dst = reinterpret_cast<uint4*>(out) + q0 * nvec;
    const int total = r.rows * nvec, live = r.live * nvec;
    copy_vectors(dst, src, live, lane);
    for (int v = live + lane; v < total; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
  }
}

// out[off_b + t] = padded[b, t] for t < min(N_b, L): runs of padded rows, like
// pad_kernel, so that no row needs an image search.  Rows of an image longer
// than L are left untouched and reported.
__global__ void __launch_bounds__(kThreads) unpad_kernel(const uint8_t* __restrict__ padded, int batch,
                                                         int64_t max_len, const int64_t* __restrict__ offsets,
                                                         int64_t rows, int nvec, int per_warp,
                                                         uint8_t* __restrict__ out, int32_t* status) {
  wait_for_previous_grid();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * kThreads) >> 5;
  const int64_t per_image = (max_len + per_warp - 1) / per_warp, runs = batch * per_image;
  for (int64_t run = warp; run < runs; run += nwarps) {
    const Run r = locate_run(run, per_image, per_warp, max_len, offsets, rows);
    if (r.first == 0 && lane == 0 && r.length > max_len) report(status, MPM_ERR_DEVICE_CHECK, r.image);
    const uint4* src = reinterpret_cast<const uint4*>(padded) + (r.image * max_len + r.first) * nvec;
    uint4* dst = reinterpret_cast<uint4*>(out) + (r.packed + r.first) * nvec;
    copy_vectors(dst, src, r.live * nvec, lane);
  }
}

int pad_grid(int num_sms, int per_sm) { return (num_sms > 0 ? num_sms : 1) * per_sm; }

// Rows of `nvec` vectors per run: the fewest (at most 32, a lane serves each
// row's mask) whose vectors fill at least nine tenths of a warp's passes of
// 32 kVecs, else those that fill them best.  Both copies of 64 images of up to
// 877 rows of 1.5 KiB take 52.7 us with 2 rows a run, 54.0 with 8; of 30
// images of up to 2000 rows of 1 KiB 33.6 with 3 rows, 35.4 with 4.  (Rows of
// 2 KiB are the one length without a gain: 36.9 us by threes, 36.1 one by one
// with 4 vectors a lane.)
int rows_per_run(int nvec) {
  constexpr int kPass = 32 * kVecs;
  int best = 1;
  double best_fill = 0;
  for (int m = 1; m <= 32 && best_fill < 0.9; ++m) {
    const int64_t vecs = static_cast<int64_t>(m) * nvec, passes = (vecs + kPass - 1) / kPass;
    const double fill = static_cast<double>(vecs) / static_cast<double>(passes * kPass);
    if (fill > best_fill) {
      best = m;
      best_fill = fill;
    }
  }
  return best;
}

// Blocks and rows per run: whole runs as long as they keep every warp busy,
// shorter ones below that.  Without rows (max_len = 0) one block still writes
// the statistics.
struct PadShape {
  int grid, per_warp;
};
PadShape pad_shape(int batch, int64_t max_len, int nvec, int wave) {
  const int64_t rows = static_cast<int64_t>(batch) * max_len, warps = static_cast<int64_t>(wave) * (kThreads / 32);
  if (rows == 0) return {1, 1};
  const int64_t even = (rows + warps - 1) / warps;
  const int most = rows_per_run(nvec);
  const int per_warp = even < most ? static_cast<int>(even) : most;
  const int64_t blocks = (rows + per_warp * (kThreads / 32) - 1) / (per_warp * (kThreads / 32));
  return {static_cast<int>(blocks < wave ? blocks : wave), per_warp};
}

}  // namespace

cudaError_t launch_pad(const void* tokens, const int64_t* offsets, int batch, int64_t rows, int64_t max_len,
                       int dim, bool bf16, void* out, uint8_t* mask, int64_t* stats, int32_t* status, int num_sms,
                       cudaStream_t stream) {
  const int nvec = dim * (bf16 ? 2 : 4) >> 4;
  static const int per_sm = resident_per_sm(pad_kernel, kThreads, 8);
  const PadShape g = pad_shape(batch, max_len, nvec, pad_grid(num_sms, per_sm));
  return launch_dependent(pad_kernel, dim3(g.grid), dim3(kThreads), 0, stream, static_cast<const uint8_t*>(tokens),
                          offsets, batch, rows, max_len, nvec, g.per_warp, static_cast<uint8_t*>(out), mask, stats,
                          status);
}

cudaError_t launch_unpad(const void* padded, int batch, int64_t max_len, const int64_t* offsets, int64_t rows,
                         int dim, bool bf16, void* out, int32_t* status, int num_sms, cudaStream_t stream) {
  const int nvec = dim * (bf16 ? 2 : 4) >> 4;
  static const int per_sm = resident_per_sm(unpad_kernel, kThreads, 8);
  const PadShape g = pad_shape(batch, max_len, nvec, pad_grid(num_sms, per_sm));
  return launch_dependent(unpad_kernel, dim3(g.grid), dim3(kThreads), 0, stream, static_cast<const uint8_t*>(padded),
                          batch, max_len, offsets, rows, nvec, g.per_warp, static_cast<uint8_t*>(out), status);
}

}  // namespace mpm
