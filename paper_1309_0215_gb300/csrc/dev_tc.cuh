// Device code shared by the tensor-core distance passes of k-means
// (k_kmeans_tc.cu: centroids resident in shared memory; k_kmeans_wide.cu:
// centroids streamed): tcgen05 primitives, the split of FP32 values into
// BF16 operands, sortable distance keys and the entries of the near-tie lists.
#pragma once
#include <cuda_bf16.h>

#include "dev_pipe.cuh"
#include "mr_internal.h"

namespace mrgb {
namespace tc {

constexpr int TM = 128;          // points per tile = MMA M = TMEM lanes
constexpr int KD = 64;           // dimensions per operand tile: one 128-byte row of BF16
constexpr int NMAX = 256;        // centroids per accumulator: MMA N
constexpr int QUARTERS = 4;      // column quarters of an accumulator, one epilogue warp each per lane quadrant
constexpr int EPI_COLS = NMAX / QUARTERS;  // at most 64 columns per epilogue warp
constexpr int GRID = 8;           // a quarter's columns as GRID x GRID: column j in row j / GRID, column j mod GRID
static_assert(GRID * GRID == EPI_COLS, "grid of a column quarter");
constexpr int CHUNK = 16;         // TMEM columns per tcgen05.ld in the epilogue

using namespace pipe;

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::f16: BF16 A and B (K-major), FP32 D, M = 128.
__host__ __device__ constexpr uint32_t mma_idesc(uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(b))
               : "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Sortable key of a distance: its FP32 bit pattern with the low 8 mantissa
// bits replaced by the centroid column, compared as a signed integer.  For
// non-negative floats the pattern is monotonic, so keys order by distance
// truncated to 16 mantissa bits (an under-statement of less than 2^-15 of
// it), then by column; a negative distance (only rounding of a point lying on
// a centroid produces one) orders below every non-negative one, and a point
// whose smallest key is negative is always re-checked.
__device__ __forceinline__ int dist_key(float dist, uint32_t col) {
  return (int)((__float_as_uint(dist) & 0xFFFFFF00u) | col);
}
__device__ __forceinline__ float key_dist(int key) { return __uint_as_float((uint32_t)key & 0xFFFFFF00u); }

// Key of a column that holds no centroid: above every finite distance's key,
// and it decodes to +inf.
constexpr int KEY_NONE = 0x7F8000FF;

// Smallest two of two sorted pairs.
__device__ __forceinline__ void top2_merge(int& a1, int& a2, int b1, int b2) {
  const int c2 = min(max(a1, b1), min(a2, b2));
  a1 = min(a1, b1);
  a2 = c2;
}

// Distances of one point to the centroids of a quarter's columns (cols of them, a
// multiple of CHUNK, from TMEM address ta on) as keys (columns counted within the
// quarter), as the minima over the columns and the rows of the quarter's grid:
// col[j mod GRID], row[j / GRID].  Any two columns differ in their grid column or
// row, so the smallest two keys are among these minima (top2_grid), at one
// three-way minimum per key where a running top-2 takes three minima and maxima.
// cn: the columns' centroid norms, infinite for columns without a centroid (the
// padding up to a multiple of 16, whose operands are zero); no other column is
// read.  sums: null, or where the columns' raw sums go.
__device__ __forceinline__ void quarter_keys(uint32_t ta, uint32_t cols, float nxv, const float* cn, int (&col)[GRID],
                                             int (&row)[GRID], float* sums = nullptr) {
  unsigned long long nx2, m2;
  asm("mov.b64 %0, {%1, %1};" : "=l"(nx2) : "f"(nxv));
  asm("mov.b64 %0, {%1, %1};" : "=l"(m2) : "f"(-2.f));
  static_assert(CHUNK == 2 * GRID, "two grid rows per load");
#pragma unroll
  for (int c = 0; c < EPI_COLS / CHUNK; ++c) {
    if ((uint32_t)(c * CHUNK) >= cols) {
      row[2 * c] = row[2 * c + 1] = KEY_NONE;
      continue;
    }
    uint32_t acc[CHUNK];
    tmem_ld(ta + c * CHUNK, acc);
    int key[CHUNK];
#pragma unroll
    for (int j = 0; j < CHUNK; j += 2) {
      unsigned long long t;
      asm("mov.b64 %0, {%1, %2};" : "=l"(t) : "r"(acc[j]), "r"(acc[j + 1]));
      const unsigned long long c2 = *reinterpret_cast<const unsigned long long*>(cn + c * CHUNK + j);
      asm("fma.rn.f32x2 %0, %1, %0, %2;" : "+l"(t) : "l"(m2), "l"(nx2));
      asm("add.rn.f32x2 %0, %0, %1;" : "+l"(t) : "l"(c2));
      float d0, d1;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(t));
      key[j] = dist_key(d0, c * CHUNK + j);
      key[j + 1] = dist_key(d1, c * CHUNK + j + 1);
    }
    if (sums)
      for (int j = 0; j < CHUNK; ++j) sums[c * CHUNK + j] = __uint_as_float(acc[j]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int* k = key + h * GRID;
      row[2 * c + h] = min(__vimin3_s32(__vimin3_s32(k[0], k[1], k[2]), k[3], k[4]), __vimin3_s32(k[5], k[6], k[7]));
    }
#pragma unroll
    for (int i = 0; i < GRID; ++i)
      col[i] = c == 0 ? min(key[i], key[GRID + i]) : __vimin3_s32(col[i], key[i], key[GRID + i]);
  }
}

// The smallest two of GRID keys.
__device__ __forceinline__ void top2_of(const int (&v)[GRID], int& w1, int& w2) {
  int lo[GRID / 2], hi[GRID / 2];
#pragma unroll
  for (int i = 0; i < GRID / 2; ++i) lo[i] = min(v[2 * i], v[2 * i + 1]), hi[i] = max(v[2 * i], v[2 * i + 1]);
#pragma unroll
  for (int w = GRID / 4; w; w >>= 1)
#pragma unroll
    for (int i = 0; i < w; ++i) {
      hi[i] = __vimin3_s32(max(lo[i], lo[i + w]), hi[i], hi[i + w]);
      lo[i] = min(lo[i], lo[i + w]);
    }
  w1 = lo[0];
  w2 = hi[0];
}

// A quarter's two smallest keys (w1, w2) from its grid's minima, their columns
// counted from c_lo on, and a lower bound lb of its other keys, but for those
// that may hide behind both in the grid (hidden_cols).  Keys above KEY_NONE
// (NaN distances) count as KEY_NONE.  lb is meaningless when w1 < 0.
__device__ __forceinline__ void top2_grid(const int (&col)[GRID], const int (&row)[GRID], uint32_t c_lo, int& w1,
                                          int& w2, int& lb) {
  int r1, r2;
  top2_of(col, w1, w2);
  top2_of(row, r1, r2);  // r1 == w1
  w1 = min(w1, KEY_NONE);
  w2 = __vimin3_s32(w2, r2, KEY_NONE);
  // the smallest minimum above w2: as distances from it, w1 and w2 wrap around
  // to the top
  uint32_t m = 0xFFFFFFFFu;
#pragma unroll
  for (int i = 0; i < GRID; ++i)
    m = __vimin3_u32(m, (uint32_t)col[i] - (uint32_t)w2 - 1u, (uint32_t)row[i] - (uint32_t)w2 - 1u);
  lb = w2 == KEY_NONE ? KEY_NONE : min((int)(m + (uint32_t)w2 + 1u), KEY_NONE);
  w1 += w1 == KEY_NONE ? 0 : (int)c_lo;
  w2 += w2 == KEY_NONE ? 0 : (int)c_lo;
}

// The two columns whose keys the minima of a quarter that starts at column c_lo
// may hide behind the keys of its columns c1 and c2, where those differ in grid
// row and grid column.
__device__ __forceinline__ bool hidden_cols(uint32_t c1, uint32_t c2, uint32_t c_lo, uint32_t& h1, uint32_t& h2) {
  constexpr uint32_t IN = GRID - 1;
  const uint32_t a = c1 - c_lo, b = c2 - c_lo;
  h1 = c_lo + ((a & ~IN) | (b & IN));
  h2 = c_lo + ((b & ~IN) | (a & IN));
  return ((a ^ b) & IN) && ((a ^ b) & ~IN);
}

// Columns of each quarter of an accumulator with cols columns (the last ones may
// have fewer): the quarters share few centroids evenly.
__device__ __forceinline__ uint32_t quarter_cols(uint32_t cols) {
  return (cols + QUARTERS * CHUNK - 1) / (QUARTERS * CHUNK) * CHUNK;
}

// BF16 hi/lo split of two values, packed little-endian (element 0 low half).
// (one paired round-to-nearest conversion for each of hi and lo)
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Byte offset of 16-byte chunk c of row r in a 128-byte-swizzled tile whose
// base is 1024-byte aligned (chunk index XOR row mod 8).
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// Centroid operands in global memory, for passes that stream them: 32 KiB
// tiles of up to NMAX centroids x KD dimensions in the swizzled layout, the
// hi and then the lo part of each (centroid chunk, dimension chunk).
constexpr uint32_t OP_TILE = NMAX * 128;
__host__ __device__ constexpr uint32_t dim_chunks(uint32_t d) { return (d + KD - 1) / KD; }
__host__ __device__ constexpr uint32_t cent_chunks(uint32_t k) { return (k + NMAX - 1) / NMAX; }
__device__ __forceinline__ void put_operand(uint8_t* bop, uint32_t d, uint32_t k, uint32_t j, float v) {
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
  uint8_t* t = bop + (uint64_t)((k / NMAX) * dim_chunks(d) + j / KD) * 2 * OP_TILE +
               swz((int)(k % NMAX), (int)((j % KD) >> 3)) + (j & 7) * 2;
  *reinterpret_cast<__nv_bfloat16*>(t) = hi;
  *reinterpret_cast<__nv_bfloat16*>(t + OP_TILE) = lo;
}

// Whether the distance pass takes the filter's list (its rows are gathered) or
// all points (whole tiles in one copy): the line is the list's extra cost.
__device__ __forceinline__ bool km_use_list(uint32_t nact, uint32_t n) { return nact < n - n / 8; }

// Append one entry per lane with `on` to a list, the warp's entries together;
// put(slot) writes it.  All 32 lanes call this.
template <class F>
__device__ __forceinline__ void warp_append(bool on, uint32_t* count, int lane, F&& put) {
  const unsigned m = __ballot_sync(0xffffffffu, on);
  if (!m) return;
  uint32_t base = 0;
  if (lane == 0) base = atomicAdd(count, (uint32_t)__popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (on) put(base + __popc(m & ((1u << lane) - 1)));
}

}  // namespace tc
}  // namespace mrgb
