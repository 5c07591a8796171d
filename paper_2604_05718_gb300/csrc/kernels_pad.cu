// Padded batches for dense-attention consumers (Section 4, Analyses: the
// images of a batch are padded to the longest merged sequence and the
// padding is masked out).  pad_kernel writes [batch, L, dim] from the packed
// rows plus a key mask and the batch's N_b statistics; unpad_kernel is the
// inverse.  Both are bandwidth-bound copies of 16-byte vectors.  A warp takes
// one row, or, where rows are short and there are enough of them, a run of rows
// of one image, contiguous on both sides, as one sequence of vectors (the rule
// is at pad_shape).  With a row a warp at every length, most lanes of short rows
// were idle: both copies of 1000 images of up to 300 rows of 64 bf16 took 103.6
// us and take 29.0, of 256 images of up to 256 rows of 384 32.8 and 31.3, of 64
// images of up to 877 rows of 768 53.5 and 52.7.
#include "mpm.h"
#include "common.cuh"
#include "launch.h"

namespace mpm {
namespace {

constexpr int kThreads = 256;
constexpr int kVecs = 6;  // 16-byte vectors in flight per lane in runs (4: 52.7 -> 53.2 us for 64 x 877 x 768, 12: 53.8)
__device__ __forceinline__ int64_t clamp_off(int64_t v, int64_t rows) { return v < 0 ? 0 : (v > rows ? rows : v); }

// A run of up to `per_warp` consecutive rows of one padded image (one row
// without RUNS): its source and destination are both contiguous.
struct Run {
  int image;
  int64_t first;   // first padded row of the run within its image
  int64_t packed;  // the image's first packed row
  int64_t length;  // the image's packed rows
  int rows, live;  // padded rows of the run, and those of them that hold tokens
};
template <bool RUNS>
__device__ __forceinline__ Run locate_run(int64_t run, int64_t per_image, int per_warp, int64_t max_len,
                                          const int64_t* __restrict__ offsets, int64_t rows) {
  Run r;
  // The short 32-bit division where it is enough.
  r.image = ((run | per_image) >> 32) == 0
                ? static_cast<int>(static_cast<uint32_t>(run) / static_cast<uint32_t>(per_image))
                : static_cast<int>(run / per_image);
  r.first = (run - r.image * per_image) * (RUNS ? per_warp : 1);
  r.packed = clamp_off(__ldg(offsets + r.image), rows);
  r.length = clamp_off(__ldg(offsets + r.image + 1), rows) - r.packed;
  const int64_t left = r.length - r.first;
  if (!RUNS) {
    r.rows = 1;
    r.live = left > 0 ? 1 : 0;
    return r;
  }
  r.rows = static_cast<int>(max_len - r.first < per_warp ? max_len - r.first : per_warp);
  r.live = static_cast<int>(left < 0 ? 0 : left < r.rows ? left : r.rows);
  return r;
}

// dst[0 .. n) = src[0 .. n), by one warp.
template <int VECS>
__device__ __forceinline__ void copy_vectors(uint4* __restrict__ dst, const uint4* __restrict__ src, int n, int lane) {
  for (int v0 = lane; v0 < n; v0 += 32 * VECS) {
    uint4 val[VECS];
#pragma unroll
    for (int u = 0; u < VECS; ++u)
      if (v0 + 32 * u < n) val[u] = __ldg(src + v0 + 32 * u);
#pragma unroll
    for (int u = 0; u < VECS; ++u)
      if (v0 + 32 * u < n) dst[v0 + 32 * u] = val[u];
  }
}

// out[b, t] = tokens[off_b + t] for t < min(N_b, L), zero rows after;
// mask[b, t] = 1 for the copied rows.  Block 0 also reduces N_b to
// (min, max, total) into stats.  An image longer than L is cut and reported.
template <int VECS, bool RUNS>
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
  const int64_t per_image = RUNS ? (max_len + per_warp - 1) / per_warp : max_len, runs = batch * per_image;
  for (int64_t run = warp; run < runs; run += nwarps) {
    const Run r = locate_run<RUNS>(run, per_image, per_warp, max_len, offsets, rows);
    if (r.first == 0 && lane == 0 && r.length > max_len) report(status, MPM_ERR_DEVICE_CHECK, r.image);
    const int64_t q0 = r.image * max_len + r.first;
    if (mask != nullptr && lane < r.rows) mask[q0 + lane] = lane < r.live ? 1 : 0;
    const uint4* src = reinterpret_cast<const uint4*>(tokens) + (r.packed + r.first) * nvec;
    uint4* dst = reinterpret_cast<uint4*>(out) + q0 * nvec;
    const int total = r.rows * nvec, live = r.live * nvec;
    copy_vectors<VECS>(dst, src, live, lane);
    for (int v = live + lane; v < total; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
  }
}

// out[off_b + t] = padded[b, t] for t < min(N_b, L): runs of padded rows, like
// pad_kernel, so that no row needs an image search.  Rows of an image longer
// than L are left untouched and reported.
template <int VECS, bool RUNS>
__global__ void __launch_bounds__(kThreads) unpad_kernel(const uint8_t* __restrict__ padded, int batch,
                                                         int64_t max_len, const int64_t* __restrict__ offsets,
                                                         int64_t rows, int nvec, int per_warp,
                                                         uint8_t* __restrict__ out, int32_t* status) {
  wait_for_previous_grid();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * kThreads) >> 5;
  const int64_t per_image = RUNS ? (max_len + per_warp - 1) / per_warp : max_len, runs = batch * per_image;
  for (int64_t run = warp; run < runs; run += nwarps) {
    const Run r = locate_run<RUNS>(run, per_image, per_warp, max_len, offsets, rows);
    if (r.first == 0 && lane == 0 && r.length > max_len) report(status, MPM_ERR_DEVICE_CHECK, r.image);
    const uint4* src = reinterpret_cast<const uint4*>(padded) + (r.image * max_len + r.first) * nvec;
    uint4* dst = reinterpret_cast<uint4*>(out) + (r.packed + r.first) * nvec;
    copy_vectors<VECS>(dst, src, r.live * nvec, lane);
  }
}

int pad_grid(int num_sms, int per_sm) { return (num_sms > 0 ? num_sms : 1) * per_sm; }

// Rows of `nvec` vectors per run: as many as fit the fewest passes of 32 kVecs
// vectors a warp that they fill to eight tenths (at most 32 rows: a lane serves
// each row's mask).  Asked for nine tenths, runs of some lengths were up to ten
// rows long, and a middling batch left SMs idle: 6.8 x 1e6 values in rows of 640
// 5.99 us with 2 rows a run, 6.63 with 7, in rows of 448 4.84 with 3, 5.67 with
// 10.
int rows_per_run(int nvec) {
  for (int pass = 32 * kVecs, room = pass;; room += pass) {
    const int m = room / nvec < 32 ? room / nvec : 32;
    if (m == 32 || 10 * m * nvec >= 8 * room) return m;
  }
}

// Are runs worth it?  A row of up to 768 B leaves a third or more of a lane's
// slots empty: they are, unless there is hardly more than a row for each warp.
// Rows of up to 1.5 KiB gain less: from five a warp on.  Longer rows fill their
// lanes, and runs only spread them less evenly over the SMs.  Geometric means
// over pad and unpad of 1 to 60 million values, time against a row a warp with
// four vectors in flight: runs 0.27 at 128 B, 0.75 at 512 B, 0.94 at 768 B; 0.87
// to 0.97 at 896 to 1536 B with more than six rows a warp, but 1.02 to 1.11 with
// two to four; 1.02 to 1.08 at 1.6 to 2 KiB and 1.04 to 1.05 at 3 to 3.5 KiB.  From
// 2064 B on a row a warp takes six vectors: 0.88 to 0.98 of the time with four.
bool worth_runs(int64_t rows, int64_t warps, int nvec) {
  if (nvec > 96) return false;
  return nvec > 48 ? rows > 4 * warps : 4 * rows > 5 * warps;
}

// Blocks and rows per run.  Without rows (max_len = 0) one block still writes
// the statistics.
struct PadShape {
  int grid, per_warp;
};
PadShape pad_shape(int64_t rows, int wave, int most) {
  if (rows == 0) return {1, 1};
  const int64_t warps = static_cast<int64_t>(wave) * (kThreads / 32), even = (rows + warps - 1) / warps;
  const int per_warp = even < most ? static_cast<int>(even) : most;
  const int64_t blocks = (rows + per_warp * (kThreads / 32) - 1) / (per_warp * (kThreads / 32));
  return {static_cast<int>(blocks < wave ? blocks : wave), per_warp};
}

// launch(kernel, shape) with the instance and shape for `rows` padded rows:
// runs of rows, or a row a warp with as many vectors in flight as its length
// needs (four hold 2 KiB).
template <typename Launch, typename Kernel>
cudaError_t launch_rows(const Launch& launch, Kernel runs, int runs_per_sm, Kernel row4, int row4_per_sm, Kernel row6,
                        int row6_per_sm, int64_t rows, int nvec, int num_sms) {
  const int wave = pad_grid(num_sms, runs_per_sm);
  if (worth_runs(rows, static_cast<int64_t>(wave) * (kThreads / 32), nvec))
    return launch(runs, pad_shape(rows, wave, rows_per_run(nvec)));
  if (nvec <= 128) return launch(row4, pad_shape(rows, pad_grid(num_sms, row4_per_sm), 1));
  return launch(row6, pad_shape(rows, pad_grid(num_sms, row6_per_sm), 1));
}

}  // namespace

cudaError_t launch_pad(const void* tokens, const int64_t* offsets, int batch, int64_t rows, int64_t max_len,
                       int dim, bool bf16, void* out, uint8_t* mask, int64_t* stats, int32_t* status, int num_sms,
                       cudaStream_t stream) {
  const int nvec = dim * (bf16 ? 2 : 4) >> 4;
  static const int runs = resident_per_sm(pad_kernel<kVecs, true>, kThreads, 8);
  static const int row4 = resident_per_sm(pad_kernel<4, false>, kThreads, 8);
  static const int row6 = resident_per_sm(pad_kernel<6, false>, kThreads, 8);
  const auto launch = [&](auto kernel, PadShape g) {
    return launch_dependent(kernel, dim3(g.grid), dim3(kThreads), 0, stream, static_cast<const uint8_t*>(tokens),
                            offsets, batch, rows, max_len, nvec, g.per_warp, static_cast<uint8_t*>(out), mask, stats,
                            status);
  };
  return launch_rows(launch, pad_kernel<kVecs, true>, runs, pad_kernel<4, false>, row4, pad_kernel<6, false>, row6,
                     static_cast<int64_t>(batch) * max_len, nvec, num_sms);
}

cudaError_t launch_unpad(const void* padded, int batch, int64_t max_len, const int64_t* offsets, int64_t rows,
                         int dim, bool bf16, void* out, int32_t* status, int num_sms, cudaStream_t stream) {
  const int nvec = dim * (bf16 ? 2 : 4) >> 4;
  static const int runs = resident_per_sm(unpad_kernel<kVecs, true>, kThreads, 8);
  static const int row4 = resident_per_sm(unpad_kernel<4, false>, kThreads, 8);
  static const int row6 = resident_per_sm(unpad_kernel<6, false>, kThreads, 8);
  const auto launch = [&](auto kernel, PadShape g) {
    return launch_dependent(kernel, dim3(g.grid), dim3(kThreads), 0, stream, static_cast<const uint8_t*>(padded),
                            batch, max_len, offsets, rows, nvec, g.per_warp, static_cast<uint8_t*>(out), status);
  };
  return launch_rows(launch, unpad_kernel<kVecs, true>, runs, unpad_kernel<4, false>, row4, unpad_kernel<6, false>, row6,
                     static_cast<int64_t>(batch) * max_len, nvec, num_sms);
}

}  // namespace mpm
