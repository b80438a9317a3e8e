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
constexpr int EPI_COLS = NMAX / QUARTERS;  // 64 columns per epilogue warp
constexpr int NSET = 4;           // independent running top-2s per epilogue thread
constexpr int CHUNK = 32;         // TMEM columns per tcgen05.ld in the epilogue

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

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
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

// Insert key into the sorted pair (t1 <= t2): three min/max.
__device__ __forceinline__ void top2_insert(int& t1, int& t2, int key) {
  const int h = max(t1, key);
  t1 = min(t1, key);
  t2 = min(t2, h);
}

// Smallest two of two sorted pairs.
__device__ __forceinline__ void top2_merge(int& a1, int& a2, int b1, int b2) {
  const int c2 = min(max(a1, b1), min(a2, b2));
  a1 = min(a1, b1);
  a2 = c2;
}

// Distances of CHUNK columns (ch .. ch + CHUNK - 1) of one point into its
// NSET running top-2s (column j goes to set j mod NSET).  MASK: some columns
// are >= k (their TMEM words are not written by the MMA and may hold
// anything), so those keys are forced to KEY_NONE.
template <bool MASK>
__device__ __forceinline__ void top2_keys(const uint32_t (&acc)[CHUNK], uint32_t ch, float nxv, const float* cn,
                                          uint32_t k, int (&t1)[NSET], int (&t2)[NSET], float* dbg_row) {
#pragma unroll
  for (int j = 0; j < CHUNK; j += 4) {
    const float4 c4 = *reinterpret_cast<const float4*>(cn + ch + j);
    const float cv[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t kk = ch + (uint32_t)(j + e);
      const float dist = fmaf(-2.f, __uint_as_float(acc[j + e]), nxv) + cv[e];
      int key = dist_key(dist, kk);
      if (MASK) {
        if (kk >= k) key = KEY_NONE;
        else if (dbg_row) dbg_row[kk] = dist;
      }
      top2_insert(t1[(j + e) % NSET], t2[(j + e) % NSET], key);
    }
  }
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

// An epilogue thread's sets reduced to its top-2 (w1, w2) and a lower bound lb
// of all its other keys: per set, the set's smallest key that is not w1 or
// w2, or its second key when both are, which bounds the rest of that set.
__device__ __forceinline__ void top2_sets(const int (&t1)[NSET], const int (&t2)[NSET], int& w1, int& w2, int& lb) {
  w1 = t1[0];
  w2 = t2[0];
#pragma unroll
  for (int a = 1; a < NSET; ++a) top2_merge(w1, w2, t1[a], t2[a]);
  lb = KEY_NONE;
#pragma unroll
  for (int a = 0; a < NSET; ++a) lb = min(lb, (t1[a] == w1 || t1[a] == w2) ? t2[a] : t1[a]);
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
