// Arg-max candidates from one 32 x 32 block of the dot-product tile, shared
// by the tensor-core affinity kernels (affinity_tc.cu, affinity_pair.cu).
//
// A warp holds 32 rows of the tile (one row per lane, as tcgen05.ld with the
// 32x32b shape delivers them) and 32 consecutive columns c..c+31 in v[].
// Row candidates: row i scores column j by G_ij / |x_j| (sc[] holds 1/|x_j|,
// NaN outside the image so that such columns never win), kept as a running
// (best score, lowest column) per thread.  Column candidates (symmetric
// tilings, blocks above the diagonal): column j scores row i by
// G_ij / |x_i|; a float warp max gives each column's best score and a ballot
// the rows reaching it, the lowest of which wins.  Equal scores always keep
// the lowest index, and -0 counts as +0, so every tiling gives the same
// answer as scoring each row against all of its columns at once.
#pragma once

#include <stdint.h>

#include "common.cuh"
#include "ptx.cuh"

namespace mpm {

// Max of x over the 32 lanes of the warp (fp32).
__device__ __forceinline__ float warp_max_f32(float x) {
  float m;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}

// scratch: 32 uint2 per warp in shared memory (column max bits, winning lanes).
// Returns, in lane L, the packed key of column c + L's candidate from these
// 32 rows (0 when there is none); the caller merges it with atomicMax.
template <bool DIAG, bool COL>
__device__ __forceinline__ unsigned long long epilogue_chunk(const uint32_t (&v)[32], const float* sc, int c,
                                                             int jd, float& best, int& bj, float inv_i, int lane,
                                                             int row_base, int n, int col0, uint2* scratch) {
#pragma unroll
  for (int k = 0; k < 32; k += 4) {
    const float4 s4 = *reinterpret_cast<const float4*>(sc + c + k);
    const float sv[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float s = __uint_as_float(v[k + u]) * sv[u];
      if (s > best && (!DIAG || c + k + u != jd)) {
        best = s;
        bj = c + k + u;
      }
    }
  }
  if (COL) {
    // Rows outside the image only occur in an image's last row block, whose
    // column candidates (blocks above it) lie wholly outside the image and
    // are dropped by the column check below; the row check is a guard.
    const bool writer = lane == 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const float s = __uint_as_float(v[k]) * inv_i;
      const float m = warp_max_f32(s);
      const uint32_t ball = __ballot_sync(0xFFFFFFFFu, s == m);
      if (writer) scratch[k] = make_uint2(__float_as_uint(m), ball);
    }
    __syncwarp();
    const uint2 r = scratch[lane];
    __syncwarp();
    const int winner = row_base + __ffs(static_cast<int>(r.y)) - 1;
    if (r.y != 0u && winner < n && col0 + c + lane < n) return make_key(__uint_as_float(r.x), winner);
  }
  return 0ull;
}

// (a0 * b0, a1 * b1) in one instruction.
__device__ __forceinline__ void mul_f32x2(float& r0, float& r1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmul.rn.f32x2 c, a, b;\n\t"
      "mov.b64 {%0, %1}, c;\n\t}"
      : "=f"(r0), "=f"(r1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// Running row maximum over groups of eight columns: the best score, the first
// column of the group it came from, and that group's first seven scores, from
// which the column is found once at the end.  (An index per column took three
// instructions a column, groups of four take 2, of eight 1.75: vit_b step
// 202.2, 200.6 and 200.3 us, mixed 233.8, 229.4 and 228.9.)
struct RowBest {
  float top = -INFINITY;
  float s[7] = {};
  int at = -1;

  // Scores of columns c .. c + 7.  A group replaces the best only when it is
  // larger, so the lowest column wins ties; NaN scores never win.
  __device__ __forceinline__ void take(const float (&x)[8], int c) {
    float m;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(x[0]), "f"(x[1]), "f"(x[2]));
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(x[3]), "f"(x[4]));
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(x[5]), "f"(x[6]));
    m = fmaxf(m, x[7]);
    if (m > top) {
      top = m;
      at = c;
#pragma unroll
      for (int i = 0; i < 7; ++i) s[i] = x[i];
    }
  }
  // The column of the best score (-1 when there is none).
  __device__ __forceinline__ int column() const {
    int i = 7;
#pragma unroll
    for (int k = 6; k >= 0; --k)
      if (s[k] == top) i = k;
    return at < 0 ? -1 : at + i;
  }
};

// One 16-column piece of a warp's slice: row candidates into the running row
// maximum, and, with COL, the column maxima and their winning rows of these
// 16 columns into the per-warp scratch entries slot .. slot + 15.  Columns go
// in pairs, two products to an instruction and two results to a 16-byte
// store: the epilogue's issue slots and shared-memory accesses are taken from
// the tensor cores' (one store per column and single products: vit_b step
// 202.9 instead of 201.7 us with paired stores and 200.9 with both; mixed
// 237.1, 234.8 and 231.6).
template <bool DIAG, bool COL>
__device__ __forceinline__ void epilogue_piece(const uint32_t (&v)[16], const float* sc, int c, int jd, RowBest& best,
                                               float inv_i, uint2* scratch, int slot, bool writer) {
#pragma unroll
  for (int k = 0; k < 16; k += 8) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; u += 4) {
      const float4 s4 = *reinterpret_cast<const float4*>(sc + c + k + u);
      mul_f32x2(x[u], x[u + 1], __uint_as_float(v[k + u]), __uint_as_float(v[k + u + 1]), s4.x, s4.y);
      mul_f32x2(x[u + 2], x[u + 3], __uint_as_float(v[k + u + 2]), __uint_as_float(v[k + u + 3]), s4.z, s4.w);
    }
    if (DIAG) {
      // A token is no candidate of its own.  (Masking only the 32 columns that
      // hold the warp's diagonal, behind a uniform branch, was 3% slower.)
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (c + k + u == jd) x[u] = -INFINITY;
    }
    best.take(x, c + k);
  }
  if (COL) {
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      float s0, s1;
      mul_f32x2(s0, s1, __uint_as_float(v[k]), __uint_as_float(v[k + 1]), inv_i, inv_i);
      const float m0 = warp_max_f32(s0), m1 = warp_max_f32(s1);
      const uint32_t b0 = __ballot_sync(0xFFFFFFFFu, s0 == m0), b1 = __ballot_sync(0xFFFFFFFFu, s1 == m1);
      if (writer)
        *reinterpret_cast<uint4*>(scratch + slot + k) = make_uint4(__float_as_uint(m0), b0, __float_as_uint(m1), b1);
    }
  }
}

// Column candidate of tile column c + lane from the scratch entries of the
// 32 columns c .. c + 31 (0 when there is none).  `origin` is added to the
// winning row for the key: the tile's first token within its image.
__device__ __forceinline__ unsigned long long column_candidate(const uint2* scratch, int lane, int row_base, int n,
                                                               int col, int origin) {
  __syncwarp();
  const uint2 r = scratch[lane];
  __syncwarp();
  const int winner = row_base + __ffs(static_cast<int>(r.y)) - 1;
  return (r.y != 0u && winner < n && col < n) ? make_key(__uint_as_float(r.x), origin + winner) : 0ull;
}

// A warp's whole COLS-column slice of one accumulator (TMEM columns
// taddr .. taddr + COLS - 1, tile columns c0 ..), read in 16-column pieces
// with the next piece's load in flight while the current one is processed.
// The loop body covers two pieces (32 columns).  DIAG: the slice may hold the
// row's own column, jd.  colcand[h] receives the column candidate of tile
// column c0 + 32 h + lane (0 when none).
template <int COLS, bool DIAG, bool COL>
__device__ __forceinline__ void epilogue_slice(uint32_t taddr, const float* sc, int c0, int jd, float& best,
                                               int& bj, float inv_i, int lane, int row_base, int n, int col0,
                                               int origin, uint2* scratch,
                                               unsigned long long (&colcand)[COLS / 32]) {
  static_assert(COLS % 32 == 0, "slices are whole 32-column pairs of pieces");
  const bool writer = lane == 0;
  RowBest rows;
  uint32_t va[16], vb[16];
  ptx::tmem_ld_32x32b_x16(taddr, va);
  ptx::tmem_wait_ld(va);
#pragma unroll
  for (int h = 0; h < COLS / 32; ++h) {
    const int c = c0 + 32 * h;
    ptx::tmem_ld_32x32b_x16(taddr + 32 * h + 16, vb);
    epilogue_piece<DIAG, COL>(va, sc, c, jd, rows, inv_i, scratch, 0, writer);
    ptx::tmem_wait_ld(vb);
    if (h + 1 < COLS / 32) ptx::tmem_ld_32x32b_x16(taddr + 32 * h + 32, va);
    epilogue_piece<DIAG, COL>(vb, sc, c + 16, jd, rows, inv_i, scratch, 16, writer);
    if (COL) {
      const unsigned long long key = column_candidate(scratch, lane, row_base, n, col0 + c + lane, origin);
#pragma unroll
      for (int g = 0; g < COLS / 32; ++g)
        if (g == h) colcand[g] = key;
    }
    if (h + 1 < COLS / 32) ptx::tmem_wait_ld(va);
  }
  best = rows.top;
  bj = rows.column();
}

// The same slice with the 32-column loop left rolled (`steps` steps of 32
// columns), for 128-column slices, whose unrolled code is twice as long:
// the column candidate of tile column c0 + 32 h + lane goes straight to
// colkeys[32 h] (colkeys points at this lane's first column) instead of a
// register array, which would need the loop unrolled.  (Measured on vit_b:
// step 0.2051-0.2054 against 0.2069-0.2073 ms unrolled; the 64-column slices
// of the 16-warp epilogue stay unrolled, where the rolled loop was 1.4%
// slower.)
template <bool DIAG, bool COL>
__device__ __forceinline__ void epilogue_slice_rolled(uint32_t taddr, const float* sc, int c0, int jd, float& best,
                                                      int& bj, float inv_i, int lane, int row_base, int n,
                                                      int col0, int origin, uint2* scratch,
                                                      unsigned long long* colkeys, int steps) {
  const bool writer = lane == 0;
  RowBest rows;
  uint32_t va[16], vb[16];
  ptx::tmem_ld_32x32b_x16(taddr, va);
  ptx::tmem_wait_ld(va);
#pragma unroll 1
  for (int h = 0; h < steps; ++h) {
    const int c = c0 + 32 * h;
    ptx::tmem_ld_32x32b_x16(taddr + 32 * h + 16, vb);
    epilogue_piece<DIAG, COL>(va, sc, c, jd, rows, inv_i, scratch, 0, writer);
    ptx::tmem_wait_ld(vb);
    const bool more = h + 1 < steps;
    if (more) ptx::tmem_ld_32x32b_x16(taddr + 32 * h + 32, va);
    epilogue_piece<DIAG, COL>(vb, sc, c + 16, jd, rows, inv_i, scratch, 16, writer);
    if (COL) {
      const unsigned long long key = column_candidate(scratch, lane, row_base, n, col0 + c + lane, origin);
      if (key != 0ull) atomicMax(colkeys + 32 * h, key);
    }
    if (more) ptx::tmem_wait_ld(va);
  }
  best = rows.top;
  bj = rows.column();
}

}  // namespace mpm
