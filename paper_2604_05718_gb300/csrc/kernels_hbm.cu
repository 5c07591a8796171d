// Bandwidth-bound MPM kernels: row norms (Eq. 1), the mutual check and
// left-to-right representative scan (Algorithm 1 steps 4-6), the pair
// average with compaction (Eq. 2), map composition (Eq. 3) and the gather
// reconstruction (Eq. 4).  All token traffic moves in 16-byte vectors, by warps
// that take one or a few rows at a time; grids are sized from the SM count and
// the rows.
#include <math.h>

#include <type_traits>

#include "mpm.h"
#include "common.cuh"

namespace mpm {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t clamp64(int64_t v, int64_t lo, int64_t hi) {
  return v < lo ? lo : (v > hi ? hi : v);
}

// ---------------------------------------------------------------------------
// Prep: status reset, offsets sanitisation + work plan (block 0), inverse
// row norms and key reset (all other blocks).  Large batches are bound by
// HBM; small ones by the dependent loads of block 0, whose plan takes one
// pass through shared memory and no rows of its own (430 rows in 3 images: 3.0
// -> 1.3 us).
// ---------------------------------------------------------------------------
// Sanitised offsets and work plan, by one block:
//   soff[b] = min(used, max_{b' <= b} max(off[b'], 0)) with used = off[batch]
//             clamped to the rows there are: non-decreasing, in range and
//             within the rows that prep covers, whatever the caller passed
//             (violations are reported);
//   plan[b] = number of affinity tiles of the images before b.
__device__ __forceinline__ void write_plan(const int64_t* __restrict__ offsets, int batch, int64_t rows,
                                           const AffinityTile& tile, const Workspace& ws) {
  __shared__ int64_t sh[32];
  __shared__ int64_t ends[kThreads + 1];
  __shared__ int bad;
  // The first images' offsets are on their way while the block meets.
  const int tid = static_cast<int>(threadIdx.x), ahead = tid < batch ? tid : batch - 1;
  const int64_t final_offset = offsets[batch];
  int64_t raw = offsets[ahead + 1], prev = offsets[ahead];
  if (threadIdx.x == 0) {
    ws.status[0] = 0;
    ws.status[1] = 0;
    ws.status[2] = 0;
    bad = -1;
  }
  __syncthreads();
  const int64_t used = clamp64(final_offset, 0, rows);
  int64_t acc = 0;
  for (int base = 0; base < batch; base += kThreads) {
    // Image `idx`: from soff[idx], which the thread before has, to soff[idx + 1].
    const int idx = base + tid;
    int64_t end = 0;
    if (idx < batch) {
      if (base > 0) {
        raw = offsets[idx + 1];
        prev = offsets[idx];
      }
      if (raw < prev || raw > rows) atomicCAS(&bad, -1, idx + 1);
      end = clamp64(raw, 0, used);
      if (idx == 0) {
        if (prev != 0) atomicExch(&bad, 0);
        const int64_t first = clamp64(prev, 0, used);
        ends[0] = ws.soff[0] = first;
        end = end > first ? end : first;
      }
    }
    const int64_t carry = base > 0 ? ends[0] : 0;
    int64_t last;
    end = block_incl_max<int64_t>(end, sh, &last, 0);
    end = end > carry ? end : carry;
    ends[threadIdx.x + 1] = end;
    __syncthreads();
    int64_t items = 0;
    if (idx < batch) {
      ws.soff[idx + 1] = end;
      items = image_items(end - ends[threadIdx.x], tile);
    }
    int64_t total;
    const int64_t incl = block_incl_sum<int64_t>(items, sh, &total);
    if (idx < batch) ws.plan[idx] = acc + incl - items;
    acc += total;
    if (threadIdx.x == 0) ends[0] = last > carry ? last : carry;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ws.plan[batch] = acc;
    if (bad >= 0) report(ws.status, MPM_ERR_DEVICE_CHECK, bad);
  }
}

// This warp's number among the warps of `blocks` blocks, this one being
// `block`.  Few rows (spread) are dealt across the blocks, so that they use
// every SM; a whole wave numbers a block's warps consecutively, so that its
// rows lie together (dealt across, the pair average of 65536 x 768 bf16 took
// 25.4 instead of 23.6 us).
__device__ __forceinline__ int64_t warp_number(int block, int blocks, bool spread) {
  const int w = static_cast<int>(threadIdx.x >> 5);
  return spread ? static_cast<int64_t>(w) * blocks + block : static_cast<int64_t>(block) * (kThreads / 32) + w;
}

// The blocks per SM are what the untraced kernel has anyway; asked for, the
// traced library's kernels, with a few registers more, have them too.  (Without,
// its pair average of 1.5 KiB rows kept two blocks an SM instead of three, and
// its timeline said 26.4 us for what takes 22.  0 leaves a kernel as it is.)
template <int ROWS, int VECS>
__global__ void __launch_bounds__(kThreads, VECS == 4 ? 0 : 5) prep_kernel(const uint8_t* __restrict__ tokens,
                                                        const int64_t* __restrict__ offsets,
                                                        int batch, int64_t rows, int row_bytes,
                                                        bool bf16, AffinityTile tile,
                                                        Workspace ws, bool spread) {
  MPM_TRACE_BEGIN(MPM_TRACE_PREP);
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  // The affinity kernel that follows only sets up barriers and tensor memory
  // before it waits for this grid, so it may take SMs as this grid drains.
  // (The other kernels do not trigger early: blocks of a dependent grid
  // parked on SMs were measured to slow the bandwidth-bound kernels.)
  allow_next_grid();
  if (blockIdx.x == 0) {
    write_plan(offsets, batch, rows, tile, ws);
    return;
  }

  // Inverse norms of every used row, and the arg-max keys reset to "none".
  // Each warp takes ROWS consecutive rows at a time and issues all of their
  // 16-byte loads (VECS a lane and row; longer rows take more passes) before
  // reducing, to keep enough bytes in flight.
  // The sweep runs from the last row to the first: the affinity kernel
  // starts with the first images, and those are then the ones this sweep
  // left in L2 (measured: 3.5 instead of 3.8 us per tile on vit_b).
  const int64_t used = clamp64(offsets[batch], 0, rows);
  auto row_of = [used](int64_t i) { return used - 1 - i; };
  const int lane = threadIdx.x & 31;
  // The blocks after block 0 take the rows.
  const int64_t warp = warp_number(blockIdx.x - 1, gridDim.x - 1, spread);
  const int64_t nwarps = static_cast<int64_t>(gridDim.x - 1) * (kThreads / 32);
  const int nvec = row_bytes >> 4;
  for (int64_t g0 = warp * ROWS; g0 < used; g0 += nwarps * ROWS) {
    float s[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) s[r] = 0.f;
    for (int v0 = lane; v0 < nvec; v0 += 32 * VECS) {
      uint4 buf[ROWS][VECS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const uint4* src = reinterpret_cast<const uint4*>(tokens + row_of(g0 + r) * row_bytes);
#pragma unroll
        for (int u = 0; u < VECS; ++u) {
          const int v = v0 + 32 * u;
          buf[r][u] = (g0 + r < used && v < nvec) ? __ldg(src + v) : make_uint4(0, 0, 0, 0);
        }
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r)
#pragma unroll
        for (int u = 0; u < VECS; ++u) s[r] += sumsq16(buf[r][u], bf16);
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) s[r] += __shfl_xor_sync(0xFFFFFFFFu, s[r], d);
    }
    if (lane < ROWS && g0 + lane < used) {
      float mine = s[0];
#pragma unroll
      for (int r = 1; r < ROWS; ++r) mine = lane == r ? s[r] : mine;
      ws.inv_norm[row_of(g0 + lane)] = 1.0f / fmaxf(sqrtf(mine), 1e-12f);
      ws.keys[row_of(g0 + lane)] = 0ull;
    }
  }
}

// ---------------------------------------------------------------------------
// Prep of fp32 tokens for the tensor cores.  Each row is scaled by the power
// of two that brings its norm into [2^14, 2^15) and split into two fp16
// values per element, x = hi + lo with hi the fp16 rounding of x and lo that
// of x - hi: 22 significant bits, as many as a tf32 high and low part hold,
// at half the bytes, and the tensor cores take fp16 at twice the tf32 rate.
// No element exceeds fp16's range, since none exceeds its row's norm, and the
// absolute error of an element far below the norm, 2^-25, is 2^-39 of the
// norm.  Dot products scale exactly, so a row's arg max is unchanged, and
// inv_norm receives the scaled rows' inverse norms (the plain ones times the
// inverse power of two), which undo the scale in the cosines.
//
// Against fp64, the rms error of the best cosines is 0.35 (64 features) to 0.70
// (4) times that through tf32 parts, 0.64 at 768, and neither it nor the largest
// error is larger for any of 17 row lengths from 4 to 2048 and seven
// distributions (normal, clustered, heavy-tailed, offset, positive, rows of
// any scale, one feature 300 times the others): half as many accumulations, in
// an order that keeps small terms (affinity_pair.cu).
//
// Bound by HBM: 65536 rows of 768 take 201 MB in and 201 MB out, 64.6 us (the
// two fp32-sized tf32 parts took 100.2).
// ---------------------------------------------------------------------------
struct RowScale {
  float s1, s2;  // the row's scale is s1 * s2
  float inv;     // 1 / max(|x|, 1e-12) of the scaled row
};

// Rows whose sum of squares says too little: zero rows, values far out of the
// usual range, infinities and NaN.  Out of line, since ordinary rows never
// come here.
__device__ __noinline__ RowScale odd_row_scale(const uint4* src, int nvec, float sumsq) {
  const int lane = threadIdx.x & 31;
  float top = 0.f;
  bool finite = true;
  for (int v = lane; v < nvec; v += 32) {
    const uint4 q = __ldg(src + v);
    const float f[4] = {__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      finite = finite && fabsf(f[k]) <= 3.402823466e38f;
      top = fmaxf(top, fabsf(f[k]));
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, d));
  // A row with an infinity or NaN has no defined cosines: all NaN, so that it
  // never is anyone's neighbour.
  if (!__all_sync(0xFFFFFFFFu, finite))
    return {__int_as_float(0x7fc00000), 1.0f, 1.0f / fmaxf(sqrtf(sumsq), 1e-12f)};
  if (top == 0.f) return {1.0f, 1.0f, 1.0f / 1e-12f};
  // Largest element to [2^7, 2^8) for the sum of squares: the norm of at most
  // 2^14 elements stays below 2^15, and its square within fp32's range.
  const int e = 7 - ilogbf(top);
  const float s1 = scalbnf(1.0f, e / 2);
  float s2 = scalbnf(1.0f, e - e / 2);
  float s = 0.f;
  for (int v = lane; v < nvec; v += 32) {
    const uint4 q = __ldg(src + v);
    const float f[4] = {__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float x = f[k] * s1 * s2;
      s = fmaf(x, x, s);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
  // Then the norm to [2^14, 2^15), like every other row's, so that small
  // elements keep as many bits.
  const float norm = sqrtf(s);
  const int up = 14 - ilogbf(norm);
  const float inv = 1.0f / fmaxf(norm, 1e-12f * s1 * s2);
  s2 = scalbnf(s2, up);
  return {s1, s2, scalbnf(inv, -up)};
}

// May the scale of a row be taken from its sum of squares?
__device__ __forceinline__ bool ordinary_sumsq(float sumsq) { return sumsq >= 0x1p-100f && sumsq <= 0x1p100f; }
// Scale of a row from its sum of squares `sumsq` (the same in every lane).
__device__ __forceinline__ RowScale row_scale(const uint4* src, int nvec, float sumsq) {
  if (!ordinary_sumsq(sumsq)) return odd_row_scale(src, nvec, sumsq);
  const float norm = sqrtf(sumsq);
  const int e = 14 - (static_cast<int>(__float_as_uint(norm) >> 23) - 127);
  return {__uint_as_float(static_cast<uint32_t>(127 + e) << 23), 1.0f,
          1.0f / fmaxf(norm, 1e-12f) * __uint_as_float(static_cast<uint32_t>(127 - e) << 23)};
}

// ROWS rows a warp and round, VECS 16-byte vectors of each in registers; with
// one row, further vectors of a longer row are read twice.
template <int ROWS, int VECS>
__global__ void __launch_bounds__(kThreads) prep_split_kernel(const uint8_t* __restrict__ tokens,
                                                              const int64_t* __restrict__ offsets, int batch,
                                                              int64_t rows, int dim, AffinityTile tile,
                                                              Workspace ws, bool spread) {
  MPM_TRACE_BEGIN(MPM_TRACE_PREP);
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  allow_next_grid();  // as in prep_kernel
  if (blockIdx.x == 0) {
    write_plan(offsets, batch, rows, tile, ws);
    return;
  }

  const int64_t used = clamp64(offsets[batch], 0, rows);
  const int lane = threadIdx.x & 31;
  const int64_t warp = warp_number(blockIdx.x - 1, gridDim.x - 1, spread);
  const int64_t nwarps = static_cast<int64_t>(gridDim.x - 1) * (kThreads / 32);
  const int nvec = dim >> 2;
  const int stride = split_stride(dim) >> 2;  // in groups of four values; those past nvec are zeros
  for (int64_t g0 = warp * ROWS; g0 < used; g0 += nwarps * ROWS) {
    const int64_t r0 = used - 1 - g0;  // last row first, as in prep_kernel
    const uint4* const src0 = reinterpret_cast<const uint4*>(tokens) + r0 * nvec;
    uint4 buf[ROWS][VECS];
    float s[ROWS];
#pragma unroll
    for (int k = 0; k < ROWS; ++k)
#pragma unroll
      for (int u = 0; u < VECS; ++u) {
        const int v = lane + 32 * u;
        buf[k][u] = (v < nvec && g0 + k < used) ? __ldg(src0 - k * nvec + v) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
      s[k] = 0.f;
#pragma unroll
      for (int u = 0; u < VECS; ++u) s[k] += sumsq16(buf[k][u], false);
    }
    if (ROWS == 1)
      for (int v = lane + 32 * VECS; v < nvec; v += 32) s[0] += sumsq16(__ldg(src0 + v), false);
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) s[k] += __shfl_xor_sync(0xFFFFFFFFu, s[k], d);
    }
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
      if (g0 + k >= used) break;
      const int64_t r = r0 - k;
      const RowScale sc = row_scale(src0 - k * nvec, nvec, s[k]);
      uint2* hi = reinterpret_cast<uint2*>(ws.split_hi) + r * stride;
      uint2* lo = reinterpret_cast<uint2*>(ws.split_lo) + r * stride;
#pragma unroll
      for (int u = 0; u < VECS; ++u) {
        const int v = lane + 32 * u;
        if (v < stride) {
          uint2 h, l;
          split_f16(buf[k][u], sc.s1, sc.s2, h, l);
          hi[v] = h;
          lo[v] = l;
        }
      }
      if (ROWS == 1)
        for (int v = lane + 32 * VECS; v < stride; v += 32) {
          uint2 h, l;
          split_f16(v < nvec ? __ldg(src0 + v) : make_uint4(0, 0, 0, 0), sc.s1, sc.s2, h, l);
          hi[v] = h;
          lo[v] = l;
        }
      if (lane == 0) {
        ws.inv_norm[r] = sc.inv;
        ws.keys[r] = 0ull;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// fp32 rows that the fp16 parts cannot decide.  An element's parts are off by
// at most 2^-39 of its row's norm (above): a cosine by about 2^-39 as the
// errors' signs go, by 2^-39 sqrt(D) at worst.  A cosine of 2^-16 or more is
// right to 2^-23, at worst 2^-23 sqrt(D), of its size, no more than the products'
// sum loses.  A row whose best cosine is smaller (rows with a huge feature of
// their own: its other features decide, and may have lost bits or vanished)
// has its neighbour found again by fp32 products of its run's tokens.  The
// kernels that read the keys of an fp32 call do that first.  Ordinary tokens
// hardly ever come here: the best of 1000 random cosines is about 3 / sqrt(D).
//
// The check reads nothing that the kernels do not read anyway and costs 0.1 to
// 0.5 us a merge (1024 x 192: 12.8 -> 13.0 us, 64 x 1024 x 192 80.9 -> 81.2, 64 x
// 1024 x 384 117.0 -> 117.3); a kernel of its own before the scan cost 1.6 to 2.4.
// Finding a row again takes one block: 0.13 ms among 1024 x 192, 0.21 ms among
// 4096 x 768, and about as long again for each further such row.
// ---------------------------------------------------------------------------
// Is the row's best cosine too small to trust?  Its score is the cosine times
// the scaled row's norm, 2^14 to 2^15 (whatever the norm's floor makes of the row
// itself), so that this holds below 2^-16 and never above 2^-15.
__device__ __forceinline__ bool undecided(unsigned long long key) {
  return (key != 0ull) & (fabsf(key_score(key)) < 0.5f);
}
// Zero rows, whose cosines are exactly 0, need nothing: their inverse norm is
// 1e12, every other row's, scaled, at most 2^-7 or so.
__device__ __forceinline__ bool undecided(unsigned long long key, float inv_norm) {
  return undecided(key) & (inv_norm < 1e11f);
}

// Does any of the rows r0 .. r1 - 1 have an element that its parts do not hold to
// 22 bits (below 2^-17 of the norm, but not 0)?  If none has, small cosines are
// right as they are, those of one-hot rows for instance.  By a whole block.
__device__ __noinline__ bool any_cut_element(const float* __restrict__ tokens, int dim, int64_t r0, int64_t r1) {
  const int lane = threadIdx.x & 31, nvec = dim >> 2;
  const int64_t warps = blockDim.x >> 5;
  for (int64_t w0 = r0; w0 < r1; w0 += 8 * warps) {
    bool cut = false;
    const int64_t end = w0 + 8 * warps < r1 ? w0 + 8 * warps : r1;
    for (int64_t r = w0 + (threadIdx.x >> 5); r < end; r += warps) {
      const uint4* const x = reinterpret_cast<const uint4*>(tokens) + r * nvec;
      float s = 0.f, least = INFINITY;
#pragma unroll 2
      for (int v = lane; v < nvec; v += 32) {
        const uint4 q = __ldg(x + v);
        const float* f = reinterpret_cast<const float*>(&q);
        s += sumsq16(q, false);
#pragma unroll
        for (int k = 0; k < 4; ++k) least = f[k] == 0.f ? least : fminf(least, fabsf(f[k]));
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
        least = fminf(least, __shfl_xor_sync(0xFFFFFFFFu, least, d));
      }
      cut |= least < INFINITY && !(ordinary_sumsq(s) && least >= 0x1p-17f * sqrtf(s));
    }
    if (__syncthreads_or(cut)) return true;
  }
  return false;
}

// `key`, or the packed row's key found again where `redo` is set: the best of
// its run by the affinity kernel's scores, products of the scaled rows times
// the neighbour's scaled inverse norm.  Ties go to the lowest index and NaN
// never wins.  Scores are compared 2^96 times as large (at most 2^126), so that
// products of two rows' smallest features do not vanish.  Called by all threads
// of a block: one row at a time, its candidates dealt over the warps.  A score
// that is small because the best neighbour's norm is below the floor (the errors
// are as much smaller) stays as it is.
__device__ __noinline__ unsigned long long decide(bool redo, unsigned long long key, int64_t row,
                                                  const float* __restrict__ tokens, int dim, int batch, int chunk,
                                                  const int64_t* soff, const float* inv_norm) {
  __shared__ unsigned long long turn, best;  // the next row (and its thread below it); its best key
  __shared__ bool floored;
  const int lane = threadIdx.x & 31, nvec = dim >> 2;
  const auto sum = [](float s) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
    return s;
  };
  // Sums of y's squares and of its products with x, each value times s1 s2.
  const auto products = [&](const uint4* x, const uint4* y, float xs1, float xs2, float ys1, float ys2) {
    float2 r = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int v = lane; v < nvec; v += 32) {
      const uint4 p = __ldg(x + v), q = __ldg(y + v);
      const float* f = reinterpret_cast<const float*>(&p);
      const float* g = reinterpret_cast<const float*>(&q);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float w = g[k] * ys1 * ys2;
        r.x = fmaf(w, w, r.x);
        r.y = fmaf(f[k] * xs1 * xs2, w, r.y);
      }
    }
    return make_float2(sum(r.x), sum(r.y));
  };
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      turn = ~0ull;
      best = 0ull;
    }
    __syncthreads();
    const unsigned long long mine = static_cast<unsigned long long>(row) << 10 | threadIdx.x;
    if (redo) atomicMin(&turn, mine);
    __syncthreads();
    const unsigned long long now = turn;
    if (now == ~0ull) return key;
    const int64_t r = static_cast<int64_t>(now >> 10);
    const int b = find_image(soff, batch, r);
    const int64_t base = soff[b];
    const int n = static_cast<int>(soff[b + 1] - base), local = static_cast<int>(r - base);
    const int first = chunk > 0 ? (local / chunk) * chunk : 0;
    const int end = chunk > 0 && n - first > chunk ? first + chunk : n;
    if (mine == now) {
      // Without the floor, 1 / 2^15 < inv_norm.
      const float inv_j = inv_norm[base + key_index(key)];
      floored = inv_j < 0.99f * 0x1p-15f && fabsf(key_score(key)) >= 0.5f * 0x1p15f * inv_j;
    }
    __syncthreads();
    if (floored) {
      redo = redo && mine != now;
      continue;
    }
    const uint4* const rows = reinterpret_cast<const uint4*>(tokens);
    const uint4* const x = rows + r * nvec;
    const RowScale a = row_scale(x, nvec, products(x, x, 1.f, 1.f, 1.f, 1.f).x);
    unsigned long long top = 0ull;
    for (int j = first + static_cast<int>(threadIdx.x >> 5); j < end; j += static_cast<int>(blockDim.x >> 5)) {
      if (j == local) continue;
      const uint4* const y = rows + (base + j) * nvec;
      float2 p = products(x, y, a.s1 * 0x1p24f, a.s2 * 0x1p24f, 1.f, 1.f);
      float score = p.y * (0x1p48f / fmaxf(sqrtf(p.x), 1e-12f));
      if (!ordinary_sumsq(p.x)) {
        const RowScale c = odd_row_scale(y, nvec, p.x);
        p = products(x, y, a.s1 * 0x1p24f, a.s2 * 0x1p24f, c.s1, c.s2);
        score = p.y * (c.inv * 0x1p48f);
      }
      const unsigned long long k = score == score ? make_key(score, j) : 0ull;
      top = k > top ? k : top;
    }
    if (lane == 0 && top != 0ull) atomicMax(&best, top);
    __syncthreads();
    if (redo && mine == now) {
      key = best == 0ull ? 0ull : make_key(key_score(best) * 0x1p-96f, key_index(best));
      redo = false;
    }
  }
}

// ---------------------------------------------------------------------------
// Mutual check + left-to-right representative scan: a cluster of C blocks
// (C = 1, 2, 4 or 8, chosen by the launch) per image.  Every block takes a run
// of consecutive rows, up to kScanElems per thread, and the blocks exchange
// their counts through distributed shared memory, so that a run's IDs start
// where the previous run's end.  The pair average that follows turns the
// counts into out_offsets.
//
// The kernel is bound by latency, not bytes: a row costs two dependent key
// loads, and a block one barrier (two for a cluster).  One block per image,
// 1024 rows at a time and three barriers a round, took 2.8 us for one image
// of 1024 rows, 6.3 for 3136, 21.6 for 16384 and 7.6 for 24 images of up to
// 4096; now 1.4, 2.6, 3.7 and 3.2.  Offsets by the last image to finish (a
// ticket, then the counts) took 1 to 2.3 us more of every batch: 64 images of
// 1024 rows 3.7 us instead of 2.0.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanElems = 4;
constexpr int kScanMaxCluster = 8;
constexpr int kAgain = 1 << 30;  // in a block's count: its image has to be scanned again
// Images whose counts every block of the pair average adds up itself.  (Up to 256
// only: merges of 257 x 64 x 64 rows 22.4 instead of 20.3 us, of 1024 x 64 x 64
// 52.6 instead of 47.9, of 1024 x 150 x 384 116.3 instead of 106.4.)
constexpr int kStagedImages = 1024;

__device__ __forceinline__ uint32_t scan_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t scan_cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t scan_cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
// Stores v at the address `p` has in block `rank` of the cluster.
__device__ __forceinline__ void store_to_rank(int32_t* p, uint32_t rank, int32_t v) {
  uint32_t at;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(at)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// May row i of an image of n rows have neighbour j?  b(i) lies in i's chunk (the
// whole image without chunking), and only a token alone in its chunk has none.
__device__ __forceinline__ bool neighbour_ok(int j, int i, int n, int chunk) {
  const int cstart = chunk > 0 ? (i / chunk) * chunk : 0;
  const int clen = chunk > 0 ? (n - cstart < chunk ? n - cstart : chunk) : n;
  return j < 0 ? clen == 1 : j < n && j != i && j >= cstart && j - cstart < clen;
}

// One image's scan once more, by a whole block, with undecided keys found again;
// returns the number of representatives.
__device__ __noinline__ int scan_again(const float* tokens, int batch, int dim, int chunk, const int64_t* soff,
                                       const unsigned long long* keys, const float* inv_norm, int b, int32_t* out_map,
                                       int2* out_reps, int32_t* status) {
  __shared__ int32_t sh[32];
  const int64_t base = soff[b];
  const int n = static_cast<int>(soff[b + 1] - base);
  const bool cut = any_cut_element(tokens, dim, base, base + n);
  int carry = 0;
  for (int c0 = 0; c0 < n; c0 += static_cast<int>(blockDim.x)) {
    const int i = c0 + static_cast<int>(threadIdx.x);
    const bool live = i < n;
    unsigned long long key = live ? keys[base + i] : 0ull;
    key = decide(cut && live && undecided(key, inv_norm[base + i]), key, base + i, tokens, dim, batch, chunk, soff,
                 inv_norm);
    int j = key_index(key);
    if (live && !neighbour_ok(j, i, n, chunk)) {
      report(status, MPM_ERR_DEVICE_CHECK, static_cast<int32_t>(base + i));
      j = -1;
    }
    key = j >= 0 ? keys[base + j] : 0ull;
    key = decide(cut && j >= 0 && undecided(key, inv_norm[base + j]), key, base + j, tokens, dim, batch, chunk, soff,
                 inv_norm);
    if (key_index(key) != i) j = -1;
    const bool rep = live && (j < 0 || i < j);
    int total;
    const int incl = block_incl_sum<int>(rep ? 1 : 0, sh, &total);
    if (rep) {
      const int r = carry + incl - 1;
      out_map[base + i] = r;
      if (j >= 0) out_map[base + j] = r;
      out_reps[base + r] = make_int2(i, j);
    }
    carry += total;
  }
  return carry;
}

// SPLIT: fp32 tokens.  An image with an undecided key is left to its first
// block, which scans it again from the start: a call in the middle of the loop
// cost every fp32 merge 1 to 6 us in spilled registers or blocks an SM.  (One
// block an SM only where the registers of four rows a thread and a cluster ask
// for it.)
template <int ELEMS, bool CLUSTER, bool SPLIT>
__global__ void __launch_bounds__(kScanThreads, CLUSTER && ELEMS > 1 ? 0 : 2)
    mutual_compact_kernel(const float* __restrict__ tokens, int batch, int dim, int chunk, Workspace ws,
                          int32_t* __restrict__ out_map, int64_t* __restrict__ out_offsets) {
  MPM_TRACE_BEGIN(MPM_TRACE_MUTUAL);
  // Every block of the cluster runs before any stores into another's memory.
  if (CLUSTER) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  wait_for_previous_grid();
  if (CLUSTER) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  MPM_TRACE_WAITED();
  __shared__ int32_t warp_count[2][ELEMS][32];
  __shared__ int32_t block_count[2][kScanMaxCluster];
  __shared__ int32_t sh[32];
  __shared__ int is_last;
  const int rank = CLUSTER ? static_cast<int>(scan_cluster_rank()) : 0;
  const int blocks = CLUSTER ? static_cast<int>(scan_cluster_size()) : 1;
  const int b = CLUSTER ? static_cast<int>(scan_cluster_id()) : static_cast<int>(blockIdx.x);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  const int64_t base = ws.soff[b];
  const int n = static_cast<int>(ws.soff[b + 1] - base);
  const int round_rows = blocks * kScanThreads;  // rows of one element per thread
  int carry = 0, buf = 0;
  [[maybe_unused]] bool again = false;
  for (int64_t c0 = 0; c0 < n; c0 += static_cast<int64_t>(round_rows) * ELEMS, buf ^= 1) {
    const int left = n - static_cast<int>(c0);
    const int elems = left >= round_rows * ELEMS ? ELEMS : (left + round_rows - 1) / round_rows;
    const int64_t first = c0 + rank * elems * kScanThreads + static_cast<int>(threadIdx.x);
    int j[ELEMS];
    uint32_t reps[ELEMS];  // ballot of the warp's representatives
    [[maybe_unused]] bool redo = false;
#pragma unroll
    for (int e = 0; e < ELEMS; ++e) {
      const int64_t i = first + e * kScanThreads;
      const unsigned long long key = (e < elems && i < n) ? ws.keys[base + i] : 0ull;
      if (SPLIT) redo |= undecided(key);
      j[e] = key_index(key);
    }
#pragma unroll
    for (int e = 0; e < ELEMS; ++e) {
      const int i = static_cast<int>(first + e * kScanThreads);  // used only where the row exists
      bool rep = false;
      if (e < elems && first + e * kScanThreads < n) {
        if (!neighbour_ok(j[e], i, n, chunk)) {
          report(ws.status, MPM_ERR_DEVICE_CHECK, static_cast<int32_t>(base + i));
          j[e] = -1;
        }
        // (i, j) is a pair of P when b(j) = i as well (Section 3.2).
        if (j[e] >= 0) {
          const unsigned long long key = ws.keys[base + j[e]];
          if (SPLIT) redo |= undecided(key);
          if (key_index(key) != i) j[e] = -1;
        }
        rep = j[e] < 0 || i < j[e];
      }
      reps[e] = __ballot_sync(0xFFFFFFFFu, rep);
      if (lane == 0) warp_count[buf][e][warp] = __popc(reps[e]);
    }
    if constexpr (SPLIT) {
      again = __syncthreads_or(redo) != 0;
      if (!CLUSTER && again) break;
    } else {
      __syncthreads();
    }
    // Representatives of this block's run before each of this warp's elements.
    int start[ELEMS], total = 0;
#pragma unroll
    for (int e = 0; e < ELEMS; ++e) {
      if (e < elems) {
        const int mine = warp_count[buf][e][lane];
        const int incl = warp_incl_sum(mine);
        start[e] = total + __shfl_sync(0xFFFFFFFFu, incl - mine, warp);
        total += __shfl_sync(0xFFFFFFFFu, incl, 31);
      }
    }
    int run_base = carry;
    if constexpr (CLUSTER) {
      // The other blocks reach this round's barrier only after they read the
      // counts of the round before the last, which this buffer held.
      if (SPLIT && again) total |= kAgain;
      if (threadIdx.x < static_cast<unsigned>(blocks)) store_to_rank(&block_count[buf][rank], threadIdx.x, total);
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      if (SPLIT) again = false;
      for (int r = 0; r < blocks; ++r) {
        int t = block_count[buf][r];
        if (SPLIT) again |= t >= kAgain;
        if (SPLIT) t &= kAgain - 1;
        run_base += r < rank ? t : 0;
        carry += t;
      }
      if (SPLIT && again) break;
    } else {
      carry += total;
    }
#pragma unroll
    for (int e = 0; e < ELEMS; ++e) {
      if (e < elems && ((reps[e] >> lane) & 1u)) {
        const int i = static_cast<int>(first + e * kScanThreads);
        const int r = run_base + start[e] + __popc(reps[e] & below);
        out_map[base + i] = r;
        if (j[e] >= 0) out_map[base + j[e]] = r;
        ws.reps[base + r] = make_int2(i, j[e]);
      }
    }
  }
  if (rank != 0) return;
  if (SPLIT && again)
    carry = scan_again(tokens, batch, dim, chunk, ws.soff, ws.keys, ws.inv_norm, b, out_map, ws.reps, ws.status);
  if (threadIdx.x == 0) ws.count[b] = carry;
  if (batch <= kStagedImages) return;
  // More images than the pair average's blocks turn into offsets themselves:
  // the last image to finish does it for all.
  if (threadIdx.x == 0) {
    // The ticket increment releases this image's count and, in the last
    // image's block, acquires all the others' (their increments came first).
    int prev;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(prev) : "l"(ws.status + 2) : "memory");
    is_last = prev == batch - 1;
  }
  __syncthreads();
  if (!is_last) return;
  // Counts -> out_offsets.  Their sum is at most the rows, which fit 32 bits.
  int acc = 0;
  for (int c0 = 0; c0 <= batch; c0 += kScanThreads) {
    const int idx = c0 + threadIdx.x;
    const int v = idx < batch ? __ldcg(ws.count + idx) : 0;
    int total;
    const int incl = block_incl_sum<int>(v, sh, &total);
    if (idx <= batch) out_offsets[idx] = acc + incl - v;
    acc += total;
  }
  if (threadIdx.x == 0) ws.status[2] = 0;
}

// ---------------------------------------------------------------------------
// Pair average + compaction (Eq. 2): one warp per output row.
// ---------------------------------------------------------------------------
// R consecutive output rows at a time, U vectors of each in flight per lane:
// all loads of a pass are issued before any store.
template <int U, int R, bool ONE>
__global__ void __launch_bounds__(kThreads, R == 1 ? 0 : 3) pair_average_kernel(const uint8_t* __restrict__ tokens,
                                                                uint8_t* __restrict__ out,
                                                                int batch, int64_t rows, int row_bytes,
                                                                bool bf16, Workspace ws, int64_t* out_offsets,
                                                                bool spread) {
  MPM_TRACE_BEGIN(MPM_TRACE_PAIR_AVERAGE);
  // First input and output row of every image.  Each block adds the counts up
  // itself: one load and a scan, where searching finished offsets is a chain
  // of dependent loads, which is what bounds few rows.
  extern __shared__ int32_t offsets_s[];  // [2 batch + 1] when staged
  __shared__ int32_t sh[32];
  const bool staged = !ONE && batch <= kStagedImages;
  int32_t* const out_s = offsets_s;             // [batch + 1]
  int32_t* const in_s = offsets_s + batch + 1;  // [batch]
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  int64_t total = 0;
  int64_t lo = 1, hi = 0, in_base = 0;  // empty: the first row is always looked up
  if (ONE) {
    total = hi = ws.count[0];
    lo = 0;
    in_base = ws.soff[0];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      out_offsets[0] = 0;
      out_offsets[1] = total;
    }
  } else if (staged) {
    int acc = 0;
    for (int base = 0; base < batch; base += kThreads) {
      const int idx = base + static_cast<int>(threadIdx.x);
      const int v = idx < batch ? ws.count[idx] : 0;
      const int64_t in = idx < batch ? ws.soff[idx] : 0;
      int sum;
      const int incl = block_incl_sum<int>(v, sh, &sum);
      if (idx < batch) {
        in_s[idx] = static_cast<int32_t>(in);
        out_s[idx] = acc + incl - v;
      }
      acc += sum;
    }
    if (threadIdx.x == 0) out_s[batch] = acc;
    __syncthreads();
    total = acc;
    if (blockIdx.x == 0)
      for (int idx = threadIdx.x; idx <= batch; idx += kThreads) out_offsets[idx] = out_s[idx];
  } else {
    total = clamp64(out_offsets[batch], 0, rows);
  }
  const int64_t warp = warp_number(blockIdx.x, gridDim.x, spread);
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * kThreads) >> 5;
  const int lane = threadIdx.x & 31, nvec = row_bytes >> 4;
  for (int64_t t0 = warp * R; t0 < total; t0 += nwarps * R) {
    const uint4* a[R];
    const uint4* p[R];
    bool pair[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t t = t0 + r < total ? t0 + r : t0;
      if (!ONE && (t >= hi || t < lo)) {
        if (staged) {
          int b = 0, top = batch - 1;
          while (b < top) {
            const int mid = (b + top + 1) >> 1;
            if (out_s[mid] <= t) b = mid; else top = mid - 1;
          }
          lo = out_s[b];
          hi = out_s[b + 1];
          in_base = in_s[b];
        } else {
          const int b = find_image(out_offsets, batch, t);
          lo = out_offsets[b];
          hi = out_offsets[b + 1];
          in_base = ws.soff[b];
        }
      }
      const int2 rep = ws.reps[in_base + (t - lo)];
      pair[r] = rep.y >= 0;
      a[r] = reinterpret_cast<const uint4*>(tokens + (in_base + rep.x) * row_bytes);
      p[r] = reinterpret_cast<const uint4*>(tokens + (in_base + (pair[r] ? rep.y : rep.x)) * row_bytes);
    }
    uint4* dst = reinterpret_cast<uint4*>(out + t0 * row_bytes);
    for (int v0 = lane; v0 < nvec; v0 += 32 * U) {
      uint4 va[R][U], vb[R][U];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int v = v0 + 32 * u;
          if (v < nvec) {
            va[r][u] = __ldcs(a[r] + v);
            if (pair[r]) vb[r][u] = __ldcs(p[r] + v);
          }
        }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int v = v0 + 32 * u;
          if (v < nvec && t0 + r < total)
            dst[static_cast<int64_t>(r) * nvec + v] = pair[r] ? avg16(va[r][u], vb[r][u], bf16) : va[r][u];
        }
    }
  }
}

// ---------------------------------------------------------------------------
// Mutual check, compaction and pair average of a small batch in one launch.
// Every block repeats the whole scan in shared memory, keeps the list of
// output rows and writes its share of them; block 0 also writes the map and
// the offsets.  Up to 1024 rows, four per thread, the scan costs less than
// the launch (1.6 us of the host) and the kernel boundary that it saves: a
// pass of two merges of 430 rows takes 28.4 us instead of 33.8, one merge of
// 1024 rows of 768 B 18.7 instead of 21.4.
// ---------------------------------------------------------------------------
constexpr int kTailElems = 4;
constexpr int kTailRows = kTailElems * kThreads;
constexpr int kTailImages = kThreads;

// Output row t: input row `first`, averaged with input row `second` if it is
// a pair (otherwise second = first).  All loads of a pass are issued before
// any store.
template <int U>
__device__ __forceinline__ void average_row(const uint8_t* __restrict__ tokens, uint8_t* __restrict__ out,
                                            int64_t first, int64_t second, bool pair, int64_t t, int row_bytes,
                                            bool bf16) {
  const int lane = threadIdx.x & 31, nvec = row_bytes >> 4;
  const uint4* a = reinterpret_cast<const uint4*>(tokens + first * row_bytes);
  const uint4* p = reinterpret_cast<const uint4*>(tokens + second * row_bytes);
  uint4* dst = reinterpret_cast<uint4*>(out + t * row_bytes);
  for (int v0 = lane; v0 < nvec; v0 += 32 * U) {
    uint4 va[U], vb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int v = v0 + 32 * u;
      if (v < nvec) {
        va[u] = __ldcs(a + v);
        if (pair) vb[u] = __ldcs(p + v);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int v = v0 + 32 * u;
      if (v < nvec) dst[v] = pair ? avg16(va[u], vb[u], bf16) : va[u];
    }
  }
}

// SPLIT: fp32 tokens, whose keys decide() checks first.
template <bool SPLIT>
__global__ void __launch_bounds__(kThreads) merge_tail_kernel(const uint8_t* __restrict__ tokens,
                                                              uint8_t* __restrict__ out, int batch, int rows,
                                                              int chunk, int row_bytes, bool bf16, Workspace ws,
                                                              int32_t* __restrict__ out_map,
                                                              int64_t* __restrict__ out_offsets) {
  __shared__ int32_t first_s[kTailImages + 1];   // first input row of every image
  __shared__ int32_t start_s[kTailImages + 1];   // first output row of every image
  __shared__ int32_t nn_s[kTailRows];            // neighbour's packed row, -1 = none; later the output row
  __shared__ uint32_t list_s[kTailRows];         // output row: input row, partner's row (0xFFFF = none) above it
  __shared__ int32_t warp_count[32];
  static_assert(kTailElems * (kThreads / 32) == 32 && kTailRows <= 0xFFFF, "one warp scans the counts; 16-bit rows");
  MPM_TRACE_BEGIN(MPM_TRACE_MUTUAL);
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  int j[kTailElems], image[kTailElems];
  [[maybe_unused]] bool redo = false;
  // Rows of the capacity past the last image have no keys of this call.
  [[maybe_unused]] const int64_t used_rows = SPLIT ? ws.soff[batch] : 0;
#pragma unroll
  for (int e = 0; e < kTailElems; ++e) {
    const int i = e * kThreads + tid;
    const unsigned long long key = i < rows ? ws.keys[i] : 0ull;
    if (SPLIT) redo |= undecided(key) & (i < used_rows);
    j[e] = key_index(key);
  }
  for (int idx = tid; idx <= batch; idx += kThreads) first_s[idx] = static_cast<int32_t>(ws.soff[idx]);
  bool some = false;
  if (SPLIT) some = __syncthreads_or(redo); else __syncthreads();
  const int lead = first_s[0], used = first_s[batch];  // rows before the first image belong to none
  if (SPLIT && some) {
    if (blockIdx.x != 0) return;  // rare: one block does it all, so that none repeats the search
    const bool cut = any_cut_element(reinterpret_cast<const float*>(tokens), row_bytes >> 2, lead, used);
    for (int e = 0; e < kTailElems; ++e) {
      const int i = e * kThreads + tid;
      const bool live = i >= lead && i < used;
      const unsigned long long key = live ? ws.keys[i] : 0ull;
      const int again = key_index(decide(cut && live && undecided(key, ws.inv_norm[i]), key, i,
                                         reinterpret_cast<const float*>(tokens), row_bytes >> 2, batch, chunk, ws.soff,
                                         ws.inv_norm));
#pragma unroll
      for (int k = 0; k < kTailElems; ++k) j[k] = k == e && live ? again : j[k];
    }
  }
#pragma unroll
  for (int e = 0; e < kTailElems; ++e) {
    const int i = e * kThreads + tid;
    int b = 0, top = batch - 1;
    while (b < top) {
      const int mid = (b + top + 1) >> 1;
      if (first_s[mid] <= i) b = mid; else top = mid - 1;
    }
    image[e] = b;
    const int base = first_s[b], n = first_s[b + 1] - base, local = i - base;
    int nn = -1;
    if (i >= lead && i < used) {
      if (!neighbour_ok(j[e], local, n, chunk)) {
        if (blockIdx.x == 0) report(ws.status, MPM_ERR_DEVICE_CHECK, i);
      } else if (j[e] >= 0) {
        nn = base + j[e];
      }
    }
    nn_s[i] = nn;
  }
  __syncthreads();
  uint32_t reps[kTailElems];
#pragma unroll
  for (int e = 0; e < kTailElems; ++e) {
    const int i = e * kThreads + tid;
    const int p = nn_s[i];
    j[e] = p >= 0 && nn_s[p] == i ? p : -1;  // the pair's other row
    reps[e] = __ballot_sync(0xFFFFFFFFu, i >= lead && i < used && (j[e] < 0 || i < j[e]));
    if (lane == 0) warp_count[e * (kThreads / 32) + warp] = __popc(reps[e]);
  }
  __syncthreads();
  const int mine = warp_count[lane];
  const int incl = warp_incl_sum(mine);
  const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
#pragma unroll
  for (int e = 0; e < kTailElems; ++e) {
    const int i = e * kThreads + tid;
    const int start = __shfl_sync(0xFFFFFFFFu, incl - mine, e * (kThreads / 32) + warp);
    if ((reps[e] >> lane) & 1u) {
      const int r = start + __popc(reps[e] & ((1u << lane) - 1u));
      nn_s[i] = r;
      if (j[e] >= 0) nn_s[j[e]] = r;
      list_s[r] = static_cast<uint32_t>(i) | (static_cast<uint32_t>(j[e] < 0 ? 0xFFFF : j[e]) << 16);
    }
  }
  __syncthreads();
  const int blocks = some ? 1 : static_cast<int>(gridDim.x);
  const int64_t nwarps = static_cast<int64_t>(blocks) * (kThreads / 32);
  for (int64_t t = warp_number(blockIdx.x, blocks, true); t < total; t += nwarps) {
    const uint32_t r = list_s[t];
    const int first = static_cast<int>(r & 0xFFFFu), second = static_cast<int>(r >> 16);
    const bool pair = second != 0xFFFF;
    average_row<4>(tokens, out, first, pair ? second : first, pair, t, row_bytes, bf16);
  }
  if (blockIdx.x != 0) return;
  // An image's first row is a representative, so its output row is where the
  // image starts; images without rows start where the next one does.
  for (int idx = tid; idx <= batch; idx += kThreads) {
    const int r = first_s[idx];
    start_s[idx] = r < used ? nn_s[r] : total;
    out_offsets[idx] = start_s[idx];
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kTailElems; ++e) {
    const int i = e * kThreads + tid;
    if (i >= lead && i < used) out_map[i] = nn_s[i] - start_s[image[e]];
  }
}

// ---------------------------------------------------------------------------
// Keys -> nearest neighbour and cosine (test / diagnostics hook).
// ---------------------------------------------------------------------------
template <bool SPLIT>
__global__ void __launch_bounds__(kThreads, 4) decode_nn_kernel(const float* __restrict__ tokens, int batch, int dim,
                                                                int chunk, Workspace ws, int32_t* __restrict__ nn,
                                                                float* __restrict__ score) {
  wait_for_previous_grid();
  const int64_t used = ws.soff[batch];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
  for (int64_t b0 = static_cast<int64_t>(blockIdx.x) * kThreads; b0 < used; b0 += stride) {
    const int64_t g = b0 + threadIdx.x;
    unsigned long long k = g < used ? ws.keys[g] : 0ull;
    const float inv = g < used ? ws.inv_norm[g] : 0.f;
    if (SPLIT && __syncthreads_or(undecided(k))) {
      // The rows of all images that this block's rows belong to.
      const int64_t last = b0 + kThreads < used ? b0 + kThreads - 1 : used - 1;
      const int64_t r0 = ws.soff[find_image(ws.soff, batch, b0)], r1 = ws.soff[find_image(ws.soff, batch, last) + 1];
      if (any_cut_element(tokens, dim, r0, r1))
        k = decide(undecided(k, inv), k, g, tokens, dim, batch, chunk, ws.soff, ws.inv_norm);
    }
    if (g >= used) continue;
    nn[g] = key_index(k);
    if (score != nullptr) score[g] = k == 0ull ? -INFINITY : key_score(k) * inv;
  }
}

// ---------------------------------------------------------------------------
// Map composition (Eq. 3).
// ---------------------------------------------------------------------------
// map1 may alias out (in-place composition): each thread reads map1[p]
// before writing out[p], and no other thread touches row p.
__global__ void compose_kernel(const int32_t* map1, const int64_t* __restrict__ off0,
                               int64_t rows0, const int32_t* __restrict__ map2,
                               const int64_t* __restrict__ off1, int64_t rows1, int batch,
                               int32_t* out, int32_t* status) {
  MPM_TRACE_BEGIN(MPM_TRACE_COMPOSE);
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  const int64_t used = clamp64(off0[batch], 0, rows0);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < used; p += stride) {
    const int b = find_image(off0, batch, p);
    const int64_t lo0 = __ldg(off0 + b), hi0 = __ldg(off0 + b + 1);
    const int64_t lo1 = __ldg(off1 + b), hi1 = __ldg(off1 + b + 1);
    const int32_t m1 = map1[p];
    int32_t r = -1;
    if (p >= lo0 && p < hi0 && m1 >= 0 && m1 < hi1 - lo1 && lo1 >= 0 && lo1 + m1 < rows1) {
      r = __ldg(map2 + lo1 + m1);
    } else {
      report(status, MPM_ERR_DEVICE_CHECK, static_cast<int32_t>(p));
    }
    out[p] = r;
  }
}

// ---------------------------------------------------------------------------
// Gather reconstruction (Eq. 4), a pure copy.  A warp takes `per_warp` (at
// most kGatherRows) consecutive grid rows: lane l resolves row p0 + l (its
// image, its map entry and the source row, all independent loads across the
// lanes), then the warp copies the rows as one run of 16-byte vectors, up to U
// of them in flight per lane.  With COMPOSE the source is composed on the way
// (Eq. 3): r*(p) = map2[off1_b + map1[p]], and r* is written to out_map if
// given.
//
// Large grids are bound by HBM, small ones by the chain of dependent loads
// (offsets, maps, row), so the rows are dealt evenly over the whole GPU: 32
// rows a warp, four at a time, left 1024 rows of 192 fp32 on 32 warps (10.0
// us, now 1.4) and 36864 rows of 1024 on 1152 warps (24.5 us, now 15.7).
// Runs of 8 rows with 12 vectors in flight were the fastest on 65536 rows of
// 768 bf16 (whole step 202.4 us; 4 rows and 8 vectors 203.3, up to 32 rows
// and 8 vectors 203.6).
// ---------------------------------------------------------------------------
constexpr int kGatherVecs = 12;
constexpr int kGatherRows = 32;  // one lane resolves each row of a run

// Rows of `nvec` vectors per run, at most.  A grid that fits L2 takes runs of two
// passes of a warp's vectors, 768, for rows shorter than 512 B, and 8 rows of
// longer ones: 80 MB of rows of 128 B 17.8 us (with 8 rows 35.8), of 256 B 16.3
// (21.7), 50 MB of rows of 768 B 10.4 us (with 16 rows 11.3).  A larger one is written fastest in runs of about 200 vectors, 3 KiB: 480
// MB of rows of 1 KiB 112.9 us with 3 rows (126.8 with 8, 186.8 with 1), of 1.5 KiB
// 113.1 with 2 (127.2), of 3 KiB 111.6 with 1 (127.8).  With 8 rows everywhere, rows of
// 1, 1.25, 2 and 8 KiB were up to 6% slower there than with 32 rows a warp, four
// at a time.
int gather_rows(int64_t rows, int nvec) {
  constexpr int64_t kLarge = 120'000'000;
  int m;
  if (rows * nvec * 16 > kLarge)
    m = (200 + nvec / 2) / nvec;
  else
    m = nvec < 32 ? 2 * 32 * kGatherVecs / nvec : 8;
  return m < 1 ? 1 : m < kGatherRows ? m : kGatherRows;
}

// Quotient e / nvec for 0 <= e < 2^17 and 1 <= nvec <= 2^12 (rows of at most
// 64 KiB): magic = floor(2^31 / nvec) + 1, so the quotient is off by less than
// e / 2^31 < 1 / nvec.
struct RowDiv {
  uint32_t nvec, magic;
  __device__ __forceinline__ uint32_t operator()(uint32_t e) const {
    return static_cast<uint32_t>((static_cast<uint64_t>(e) * magic) >> 31);
  }
};
RowDiv row_div(int row_bytes) {
  const uint32_t nvec = static_cast<uint32_t>(row_bytes >> 4);
  return {nvec, nvec == 1 ? 0x80000000u : 0x80000000u / nvec + 1u};
}

// An array of offsets in global memory, or its copy in shared memory.
template <bool STAGED>
struct Offsets {
  const int64_t* p;
  __device__ __forceinline__ int64_t operator[](int k) const { return STAGED ? p[k] : __ldg(p + k); }
};

// Finds the image of row p, reusing the previous answer when p is still in
// the same image (rows are visited in increasing order by each warp).
template <bool STAGED>
struct ImageCursor {
  int b = 0;
  int64_t lo = 1, hi = 0;  // empty: forces the first search
  __device__ __forceinline__ void locate(const Offsets<STAGED>& off, int batch, int64_t p) {
    if (p >= lo && p < hi) return;
    int last = batch - 1;
    b = 0;
    while (b < last) {
      const int mid = (b + last + 1) >> 1;
      if (off[mid] <= p) b = mid; else last = mid - 1;
    }
    lo = off[b];
    hi = off[b + 1];
  }
};

// Images from which on every block copies their offsets to shared memory: a
// search in global memory is a chain of dependent loads (64 images of 1024 x
// 768 bf16: 22.9 instead of 21.6 us, 32 of 1024 x 384: 8.1 instead of 7.5),
// but for a few images the copy and its barrier take longer (3 images of 1024 x
// 384: 2.69 against 2.49 us; from 4 to 10 images the two are within 3%, 12: 3.75
// against 3.85).  The upper bound keeps the copy within 6 KiB.
constexpr int kStagedFrom = 9, kStagedTo = 256;

template <int U, bool COMPOSE, bool STAGED>
__global__ void __launch_bounds__(kThreads) gather_kernel(const uint8_t* __restrict__ merged,
                                                          const int64_t* __restrict__ moff,
                                                          int64_t merged_rows,
                                                          const int32_t* map,
                                                          const int64_t* __restrict__ goff,
                                                          int64_t grid_rows,
                                                          const int32_t* __restrict__ map2,
                                                          const int64_t* __restrict__ off1, int64_t rows1,
                                                          int32_t* out_map, int batch, RowDiv row, int per_warp,
                                                          uint8_t* __restrict__ out, int32_t* status) {
  MPM_TRACE_BEGIN(MPM_TRACE_GATHER);
  wait_for_previous_grid();
  MPM_TRACE_WAITED();
  Offsets<STAGED> grid_at{goff}, merged_at{moff}, mid_at{off1};
  if constexpr (STAGED) {
    extern __shared__ int64_t offs_s[];  // goff, moff and (COMPOSE) off1, [batch + 1] each
    for (int k = threadIdx.x; k <= batch; k += kThreads) {
      offs_s[k] = goff[k];
      offs_s[batch + 1 + k] = moff[k];
      if (COMPOSE) offs_s[2 * (batch + 1) + k] = off1[k];
    }
    __syncthreads();
    grid_at.p = offs_s;
    merged_at.p = offs_s + batch + 1;
    mid_at.p = offs_s + 2 * (batch + 1);
  }
  const int lane = threadIdx.x & 31;
  // Neighbouring runs go to neighbouring blocks, so that few rows still use
  // every SM.
  const int64_t warp = static_cast<int64_t>(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * kThreads) >> 5;
  const int64_t used = clamp64(grid_at[batch], 0, grid_rows);
  ImageCursor<STAGED> cur;
  for (int64_t p0 = warp * per_warp; p0 < used; p0 += nwarps * per_warp) {
    // Lane l resolves grid row p0 + l.
    const int64_t p = p0 + lane;
    const int nrows = static_cast<int>(used - p0 < per_warp ? used - p0 : per_warp);
    int32_t src = -1;  // merged row to copy, -1 = none (zero row)
    if (lane < nrows) {
      int32_t m = map[p];
      cur.locate(grid_at, batch, p);
      const int64_t mlo = merged_at[cur.b], mhi = merged_at[cur.b + 1];
      bool ok = p >= cur.lo && p < cur.hi;
      if (COMPOSE) {
        // Stage-1 index of this grid row, then its stage-2 (merged) index.
        const int64_t lo1 = mid_at[cur.b], hi1 = mid_at[cur.b + 1];
        ok = ok && m >= 0 && m < hi1 - lo1 && lo1 >= 0 && lo1 + m < rows1;
        m = ok ? __ldg(map2 + lo1 + m) : -1;
      }
      ok = ok && m >= 0 && m < mhi - mlo && mlo >= 0 && mlo + m < merged_rows;
      if (!ok) report(status, MPM_ERR_DEVICE_CHECK, static_cast<int32_t>(p));
      // This lane alone reads and writes entry p, so out_map may alias map.
      if (COMPOSE && out_map != nullptr) out_map[p] = ok ? m : -1;
      src = ok ? static_cast<int32_t>(mlo + m) : -1;
    }
    const uint32_t total = static_cast<uint32_t>(nrows) * row.nvec;
    uint4* dst = reinterpret_cast<uint4*>(out) + p0 * row.nvec;
    for (uint32_t e0 = lane; e0 < total + lane; e0 += 32 * U) {
      uint4 val[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t e = e0 + 32 * u;
        const uint32_t r = row(e);
        const int32_t s = __shfl_sync(0xFFFFFFFFu, src, r & 31);
        if (e < total)
          val[u] = s >= 0 ? __ldg(reinterpret_cast<const uint4*>(merged) + static_cast<int64_t>(s) * row.nvec +
                                  (e - r * row.nvec))
                          : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (e0 + 32 * u < total) __stcs(dst + e0 + 32 * u, val[u]);
    }
  }
}

int grid_for(int num_sms, int per_sm) { return (num_sms > 0 ? num_sms : 1) * per_sm; }

// Blocks for `items` rows (or pairs of rows), one per warp and round: at most
// one wave; fewer items get a block per four of them, spread over its warps'
// numbers, so that no whole wave is launched for them.
struct RowGrid {
  int blocks;
  bool spread;
};
RowGrid row_grid(int64_t items, int wave) {
  const int64_t blocks = (items + 3) / 4;
  if (blocks >= wave) return {wave, false};
  return {blocks > 1 ? static_cast<int>(blocks) : 1, true};
}

// Blocks and rows per warp for `rows` rows: at most `wave` blocks, and rows
// dealt evenly over their warps (at most `most` of up to 32 a warp and round).
struct RunShape {
  int grid, per_warp;
};
RunShape run_shape(int64_t rows, int wave, int block_warps, int most) {
  const int64_t warps = static_cast<int64_t>(wave) * block_warps;
  const int64_t rounds = (rows + most * warps - 1) / (most * warps);
  const int64_t per_warp = (rows + warps * rounds - 1) / (warps * rounds);
  const int64_t need = (rows + per_warp * block_warps - 1) / (per_warp * block_warps);
  return {static_cast<int>(need < wave ? need : wave), static_cast<int>(per_warp)};
}

}  // namespace

#ifdef MPM_TRACE
cudaError_t trace_copy_hbm(unsigned long long* out, bool reset) { return trace_table(out, reset); }
#endif

cudaError_t launch_prep(const void* tokens, const int64_t* offsets, int batch, int64_t rows, int dim,
                        bool bf16, AffinityTile tile, const Workspace& ws, int num_sms,
                        cudaStream_t stream) {
  const int row_bytes = dim * (bf16 ? 2 : 4);
  if (ws.split_hi != nullptr) {
    const auto launch = [&](auto kernel, int per_sm, int warp_rows) {
      const RowGrid g = row_grid((rows + warp_rows - 1) / warp_rows, grid_for(num_sms, per_sm) - 1);
      return launch_dependent(kernel, dim3(1 + g.blocks), dim3(kThreads), 0, stream,
                              static_cast<const uint8_t*>(tokens), offsets, batch, rows, dim, tile, ws, g.spread);
    };
    // Rows and vectors per warp and round by the row's length, in as few
    // registers as it needs.  One row and eight vectors for every length left most
    // slots of short rows empty: queries of 64-token images, 3000 of 16 features
    // 104.8 us (75.5 with 2 x 1, 82.0 with 1 x 1, 78.1 with 4 x 1), 976 of 192 features
    // 59.1 (50.0 with 2 x 2, 50.7 with 1 x 2), 488 of 384 49.2 (47.2 with 1 x 4, 48.3
    // with 2 x 4).
    if (dim <= 128) {
      static const int per_sm = resident_per_sm(prep_split_kernel<2, 1>, kThreads, 8);
      return launch(prep_split_kernel<2, 1>, per_sm, 2);
    }
    if (dim <= 256) {
      static const int per_sm = resident_per_sm(prep_split_kernel<2, 2>, kThreads, 8);
      return launch(prep_split_kernel<2, 2>, per_sm, 2);
    }
    if (dim <= 512) {
      static const int per_sm = resident_per_sm(prep_split_kernel<1, 4>, kThreads, 8);
      return launch(prep_split_kernel<1, 4>, per_sm, 1);
    }
    static const int per_sm = resident_per_sm(prep_split_kernel<1, 8>, kThreads, 8);
    return launch(prep_split_kernel<1, 8>, per_sm, 1);
  }
  // Rows and vectors per warp and round by the row's length, so that no load
  // slot is empty: with 2 x 3 for every length, rows of 2 KiB took two passes
  // (36864 of them 17.9 us, now 16.5) and rows of 768 B half the slots (32768
  // of them 8.7, now 8.0); 4 x 3 and 1 x 3 were slower for 1.5 KiB.  Rows of
  // 2 to 6 KiB take the width that their passes fill better: 3 for 1152, 1232 and
  // 2144 features (queries of 64-token images 43.1 instead of 45.2 us, 41.7
  // instead of 42.9, 39.1 instead of 40.7), 4 for 1544 and 2048 (51.9 instead of
  // 52.6, 36.6 instead of 36.9) and for longer rows (3584: 40.0 instead of 40.7).
  const int nvec = row_bytes >> 4;
  const bool three =
      nvec > 64 && (nvec <= 96 || (nvec > 128 && nvec <= 384 && (nvec + 95) / 96 * 96 <= (nvec + 127) / 128 * 128));
  const auto launch = [&](auto kernel, int per_sm, int warp_rows) {
    const RowGrid g = row_grid((rows + warp_rows - 1) / warp_rows, grid_for(num_sms, per_sm) - 1);
    return launch_dependent(kernel, dim3(1 + g.blocks), dim3(kThreads), 0, stream, static_cast<const uint8_t*>(tokens),
                            offsets, batch, rows, row_bytes, bf16, tile, ws, g.spread);
  };
  if (nvec <= 32) {
    static const int per_sm = resident_per_sm(prep_kernel<4, 1>, kThreads, 8);
    return launch(prep_kernel<4, 1>, per_sm, 4);
  }
  if (nvec <= 64) {
    static const int per_sm = resident_per_sm(prep_kernel<3, 2>, kThreads, 8);
    return launch(prep_kernel<3, 2>, per_sm, 3);
  }
  if (three) {
    static const int per_sm = resident_per_sm(prep_kernel<2, 3>, kThreads, 8);
    return launch(prep_kernel<2, 3>, per_sm, 2);
  }
  static const int per_sm = resident_per_sm(prep_kernel<2, 4>, kThreads, 8);
  return launch(prep_kernel<2, 4>, per_sm, 2);
}

cudaError_t launch_mutual_compact(const void* tokens, int batch, int64_t rows, int dim, int64_t chunk,
                                  const Workspace& ws, int32_t* out_map, int64_t* out_offsets, int num_sms,
                                  cudaStream_t stream) {
  // One block per 1024 rows of the mean image (the images' own lengths are on
  // the device), as long as all blocks run at once: two on an SM, one where the
  // mean image needs four rows per thread in a cluster (52 registers).  Longer
  // images take more rows per thread.  (With two assumed everywhere, 40 images
  // of 6000 rows took 160 blocks on 152 SMs: a merge 81.4 us, now 78.6; 100 of
  // 2500 86.4 and 82.5.)
  const int64_t mean = (rows + batch - 1) / batch;
  int blocks = 1;
  while (blocks < kScanMaxCluster && static_cast<int64_t>(blocks) * kScanThreads < mean) {
    const int per_sm = 2 * static_cast<int64_t>(blocks) * kScanThreads < mean ? 1 : 2;
    if (2 * static_cast<int64_t>(blocks) * batch > static_cast<int64_t>(per_sm) * num_sms) break;
    blocks *= 2;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(batch) * blocks);
  cfg.blockDim = dim3(kScanThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = blocks;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = blocks > 1 ? 2 : 1;
  // A chunk at least as long as the batch is the whole image.
  const int chunk32 = chunk < rows ? static_cast<int>(chunk) : 0;
  // Four rows per thread, and the cluster's barriers, only where the mean
  // image needs them: they take 1 us more on images of 1024 rows.
  const bool more = static_cast<int64_t>(blocks) * kScanThreads < mean;
  const auto pick = [&](auto split) {
    constexpr bool S = decltype(split)::value;
    return blocks > 1 ? (more ? mutual_compact_kernel<kScanElems, true, S> : mutual_compact_kernel<1, true, S>)
                      : (more ? mutual_compact_kernel<kScanElems, false, S> : mutual_compact_kernel<1, false, S>);
  };
  const auto kernel = ws.split_hi != nullptr ? pick(std::true_type{}) : pick(std::false_type{});
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<const float*>(tokens), batch, dim, chunk32, ws, out_map,
                            out_offsets);
}

cudaError_t launch_pair_average(const void* tokens, void* out_tokens, int batch, int64_t rows,
                                int dim, bool bf16, const Workspace& ws,
                                int64_t* out_offsets, int num_sms, cudaStream_t stream) {
  const int row_bytes = dim * (bf16 ? 2 : 4);
  // A single image needs no shared memory and no barriers (with them, one of
  // 3136 rows took 1 us more a merge).
  if (batch == 1) {
    static const int per_sm = resident_per_sm(pair_average_kernel<4, 1, true>, kThreads, 8);
    const RowGrid g = row_grid(rows, grid_for(num_sms, per_sm));
    return launch_dependent(pair_average_kernel<4, 1, true>, dim3(g.blocks), dim3(kThreads), 0, stream,
                            static_cast<const uint8_t*>(tokens), static_cast<uint8_t*>(out_tokens), batch, rows,
                            row_bytes, bf16, ws, out_offsets, g.spread);
  }
  const auto launch = [&](auto kernel, int per_sm, int warp_rows) {
    const RowGrid g = row_grid((rows + warp_rows - 1) / warp_rows, grid_for(num_sms, per_sm));
    const size_t smem = batch <= kStagedImages ? (2 * static_cast<size_t>(batch) + 1) * sizeof(int32_t) : 0;
    return launch_dependent(kernel, dim3(g.blocks), dim3(kThreads), smem, stream, static_cast<const uint8_t*>(tokens),
                            static_cast<uint8_t*>(out_tokens), batch, rows, row_bytes, bf16, ws, out_offsets,
                            g.spread);
  };
  // Rows and vectors per warp and round by the row's length, so that few load
  // slots are empty (1 x 4 for every length: 32768 rows of 768 B 10.4 us, by
  // twos 8.3; passes of two merges of 256 x 512 rows of 256 B 140.5 us with 2 x
  // 2, 128.6 with 4 x 1, of 64 x 1024 rows of 1.5 KiB 197.6 with 1 x 4, 196.4
  // with 2 x 3; 2 x 4 for 2 KiB was slower, 196.1 instead of 192.2).
  if (row_bytes <= 512) {
    static const int per_sm = resident_per_sm(pair_average_kernel<1, 4, false>, kThreads, 8);
    return launch(pair_average_kernel<1, 4, false>, per_sm, 4);
  }
  if (row_bytes <= 1024) {
    static const int per_sm = resident_per_sm(pair_average_kernel<2, 2, false>, kThreads, 8);
    return launch(pair_average_kernel<2, 2, false>, per_sm, 2);
  }
  if (row_bytes <= 1536) {
    static const int per_sm = resident_per_sm(pair_average_kernel<3, 2, false>, kThreads, 8);
    return launch(pair_average_kernel<3, 2, false>, per_sm, 2);
  }
  static const int per_sm = resident_per_sm(pair_average_kernel<4, 1, false>, kThreads, 8);
  return launch(pair_average_kernel<4, 1, false>, per_sm, 1);
}

bool merge_tail_fits(int batch, int64_t rows) { return rows > 0 && rows <= kTailRows && batch <= kTailImages; }

cudaError_t launch_merge_tail(const void* tokens, void* out_tokens, int batch, int64_t rows, int dim, bool bf16,
                              int64_t chunk, const Workspace& ws, int32_t* out_map, int64_t* out_offsets, int num_sms,
                              cudaStream_t stream) {
  const auto launch = [&](auto kernel, int per_sm) {
    return launch_dependent(kernel, dim3(row_grid(rows, grid_for(num_sms, per_sm)).blocks), dim3(kThreads), 0, stream,
                            static_cast<const uint8_t*>(tokens), static_cast<uint8_t*>(out_tokens), batch,
                            static_cast<int>(rows), chunk < rows ? static_cast<int>(chunk) : 0,
                            dim * (bf16 ? 2 : 4), bf16, ws, out_map, out_offsets);
  };
  if (ws.split_hi != nullptr) {
    static const int per_sm = resident_per_sm(merge_tail_kernel<true>, kThreads, 8);
    return launch(merge_tail_kernel<true>, per_sm);
  }
  static const int per_sm = resident_per_sm(merge_tail_kernel<false>, kThreads, 8);
  return launch(merge_tail_kernel<false>, per_sm);
}

cudaError_t launch_decode_nn(const void* tokens, int batch, int64_t rows, int dim, int64_t chunk, const Workspace& ws,
                             int32_t* out_nn, float* out_score, int num_sms, cudaStream_t stream) {
  const auto launch = [&](auto kernel) {
    return launch_dependent(kernel, dim3(grid_for(num_sms, 4)), dim3(kThreads), 0, stream,
                            static_cast<const float*>(tokens), batch, dim,
                            chunk < rows ? static_cast<int>(chunk) : 0, ws, out_nn, out_score);
  };
  return ws.split_hi != nullptr ? launch(decode_nn_kernel<true>) : launch(decode_nn_kernel<false>);
}

cudaError_t launch_compose(const int32_t* map1, const int64_t* off0, int64_t rows0,
                           const int32_t* map2, const int64_t* off1, int64_t rows1, int batch,
                           int32_t* out, int32_t* status, int num_sms, cudaStream_t stream) {
  return launch_dependent(compose_kernel, dim3(grid_for(num_sms, 4)), dim3(kThreads), 0, stream, map1, off0, rows0,
                          map2, off1, rows1, batch, out, status);
}

namespace {
// Gather, or composition and gather (map2 and off1 given).
template <bool COMPOSE>
cudaError_t launch_gather_kernel(const void* merged, const int64_t* moff, int64_t merged_rows, const int32_t* map,
                                 const int64_t* goff, int64_t grid_rows, const int32_t* map2, const int64_t* off1,
                                 int64_t rows1, int32_t* out_map, int batch, int dim, bool bf16, void* out,
                                 int32_t* status, int num_sms, cudaStream_t stream) {
  const int row_bytes = dim * (bf16 ? 2 : 4);
  const auto launch = [&](auto kernel, int per_sm, size_t smem) {
    const RunShape g =
        run_shape(grid_rows, grid_for(num_sms, per_sm), kThreads / 32, gather_rows(grid_rows, row_bytes >> 4));
    return launch_dependent(kernel, dim3(g.grid), dim3(kThreads), smem, stream, static_cast<const uint8_t*>(merged),
                            moff, merged_rows, map, goff, grid_rows, map2, off1, rows1, out_map, batch,
                            row_div(row_bytes), g.per_warp, static_cast<uint8_t*>(out), status);
  };
  if (batch >= kStagedFrom && batch <= kStagedTo) {
    static const int per_sm = resident_per_sm(gather_kernel<kGatherVecs, COMPOSE, true>, kThreads, 8);
    return launch(gather_kernel<kGatherVecs, COMPOSE, true>, per_sm,
                  (COMPOSE ? 3 : 2) * sizeof(int64_t) * (static_cast<size_t>(batch) + 1));
  }
  static const int per_sm = resident_per_sm(gather_kernel<kGatherVecs, COMPOSE, false>, kThreads, 8);
  return launch(gather_kernel<kGatherVecs, COMPOSE, false>, per_sm, 0);
}
}  // namespace

cudaError_t launch_gather(const void* merged, const int64_t* moff, int64_t merged_rows,
                          const int32_t* map, const int64_t* goff, int64_t grid_rows, int batch,
                          int dim, bool bf16, void* out, int32_t* status, int num_sms,
                          cudaStream_t stream) {
  return launch_gather_kernel<false>(merged, moff, merged_rows, map, goff, grid_rows, nullptr, nullptr, 0, nullptr,
                                     batch, dim, bf16, out, status, num_sms, stream);
}

cudaError_t launch_compose_gather(const void* merged, const int64_t* moff, int64_t merged_rows,
                                  const int32_t* map1, const int64_t* off0, int64_t rows0,
                                  const int32_t* map2, const int64_t* off1, int64_t rows1, int batch, int dim,
                                  bool bf16, void* out, int32_t* out_map, int32_t* status, int num_sms,
                                  cudaStream_t stream) {
  return launch_gather_kernel<true>(merged, moff, merged_rows, map1, off0, rows0, map2, off1, rows1, out_map, batch,
                                    dim, bf16, out, status, num_sms, stream);
}

}  // namespace mpm
