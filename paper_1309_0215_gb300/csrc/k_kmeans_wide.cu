// k-means distance pass on the tensor cores for shapes whose centroids do not
// stay in one SM's shared memory: 64 < D <= 256 or K > 256 (FP32 jobs).
//
// The contraction, the split of each value into two BF16 parts, the keys, the
// margin tests and their error bounds are those of k_kmeans_tc.cu; what
// differs is where the operands come from.  Per tile of 128 points:
//   * 8 converter warps write the points' hi and lo parts for all dimensions
//     (one operand tile per 64 dimensions) and ||x||^2; the tile stays while
//     every centroid passes by;
//   * one producer thread streams the centroids' operand tiles (256
//     centroids x 64 dimensions, hi then lo; made once per round by the
//     kernel that makes the centroids) from L2 through a ring with bulk
//     copies, and one thread issues the MMAs: per centroid chunk, over the
//     dimension chunks, hi.hi + lo.hi when the hi tile is there and hi.lo
//     when the lo tile is, into one of two 256-column TMEM accumulators;
//   * 16 epilogue warps reduce each accumulator to each column quarter's two
//     smallest keys and a lower bound of the others, and 2 finalizer warps keep
//     every point's KM_CAND_MAX smallest keys over all centroid chunks, and a
//     lower bound of the rest, until the last chunk decides the point.
//
// Bounds: the MMAs need 3 * 2 N K D operations, each point tile reads every
// centroid once from L2 (4 K D bytes per 128 points) and the epilogue takes
// about 7 instructions per distance.  At 250,000 x 128, K = 512 the pass
// takes 105 us; the SIMT pass, limited by the FP32 pipe and by its
// per-thread top-3 selection, took 2,130 us.  Two point tiles fit shared
// memory up to D = 128 and the conversion overlaps the MMAs; beyond that one.
#include "dev_tc.cuh"

namespace mrgb {
namespace {

using namespace tc;

constexpr int EPI_WARPS = 16;
constexpr int MMA_WARP = EPI_WARPS;
constexpr int CVT_WARP0 = MMA_WARP + 1;
constexpr int CVT_WARPS = 8;
constexpr int CVT_ROWS = TM / CVT_WARPS;  // 16: 8 steps of 2 rows
constexpr int FIN_WARP0 = CVT_WARP0 + CVT_WARPS;
constexpr int FIN_WARPS = 2;
constexpr int FIN_QUADS = 4 / FIN_WARPS;
constexpr int COPY_WARP = FIN_WARP0 + FIN_WARPS;
constexpr int WD_THREADS = (COPY_WARP + 1) * 32;  // 896
constexpr int ACCS = 2;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t DC_MAX_W = 4;        // D <= 256
constexpr uint32_t K_MAX_W = 4096;      // 12-bit candidates
constexpr uint32_t A_TILE = TM * 128;   // one operand tile of points
constexpr uint32_t OPERANDS = 192 * 1024;  // shared memory for point and centroid operands
constexpr int RING_MAX = 4, ABUF_MAX = 2;
static_assert(CVT_ROWS == 16 && EPI_WARPS == 4 * QUARTERS, "warp roles");

struct alignas(16) WideCtl {
  uint32_t xw1[ACCS][QUARTERS][TM], xw2[ACCS][QUARTERS][TM], xlb[ACCS][QUARTERS][TM];
  float xnx[ACCS][TM];
  float nx[2][TM];
  float center[DC_MAX_W * KD];
  unsigned long long full_a[ABUF_MAX], empty_a[ABUF_MAX], nx_free[2];
  unsigned long long full_b[RING_MAX], empty_b[RING_MAX];
  unsigned long long full_acc[ACCS], empty_acc[ACCS], xfull[ACCS], xfree[ACCS], drained;
  uint32_t tmem_base;
  int err;
};

// point buffers and ring stages by the number of dimension chunks
__host__ __device__ constexpr uint32_t abufs(uint32_t dc) { return dc <= 2 ? 2 : 1; }
__host__ __device__ constexpr uint32_t ring(uint32_t dc) {
  return (OPERANDS - abufs(dc) * dc * 2 * A_TILE) / OP_TILE < (uint32_t)RING_MAX
             ? (OPERANDS - abufs(dc) * dc * 2 * A_TILE) / OP_TILE
             : (uint32_t)RING_MAX;
}
inline size_t wide_smem(uint32_t k) { return 1024 + OPERANDS + sizeof(WideCtl) + (size_t)cent_chunks(k) * NMAX * 4; }
static_assert(1024 + OPERANDS + sizeof(WideCtl) + K_MAX_W * 4 <= 232448, "shared memory of one CTA");

// Insert (key, chunk) into the sorted list t; what falls out bounds the rest.
__device__ __forceinline__ void list_insert(int (&t)[KM_CAND_MAX], uint32_t (&c)[KM_CAND_MAX], int& rest, int key,
                                            uint32_t ch) {
  if (__any_sync(0xffffffffu, key < t[KM_CAND_MAX - 1])) {
#pragma unroll
    for (uint32_t i = 0; i < KM_CAND_MAX; ++i) {
      const bool lt = key < t[i];
      const int tk = lt ? t[i] : key;
      const uint32_t tc = lt ? c[i] : ch;
      t[i] = lt ? key : t[i];
      c[i] = lt ? ch : c[i];
      key = tk;
      ch = tc;
    }
  }
  rest = min(rest, key);
}

// SUMS: the sums of every point and column go to sums [tiles TM][chunks NMAX], for
// tests.
template <bool SUMS = false>
__global__ void __launch_bounds__(WD_THREADS, 1)
km_wide_assign_kernel(const float* __restrict__ x, uint32_t n, uint32_t d, uint32_t k,
                      const uint8_t* __restrict__ bop, const float* __restrict__ center,
                      const float* __restrict__ cnorm, const unsigned int* cmax_bits, uint32_t* __restrict__ assign,
                      uint32_t* nchg, uint32_t* __restrict__ list, uint32_t* nlist, KmFew* __restrict__ few,
                      uint32_t* nfew, unsigned long long* timeouts, float* sums, long long polls,
                      unsigned int* maxabs) {
  extern __shared__ uint8_t wd_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(wd_raw) + 1023) & ~uintptr_t(1023));
  WideCtl& S = *reinterpret_cast<WideCtl*>(base + OPERANDS);
  float* cn = reinterpret_cast<float*>(&S + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t dc = dim_chunks(d), nc = cent_chunks(k), nab = abufs(dc), nring = ring(dc);
  const uint32_t npad = (k + 15) & ~15u;
  const uint32_t ntiles = (n + TM - 1) / TM;
  uint8_t* ring_b = base + nab * dc * 2 * A_TILE;  // point operands first: [buffer][dim chunk][hi, lo]
  volatile int* err = &S.err;

  if (threadIdx.x == 0) {
    S.err = 0;
    for (uint32_t q = 0; q < nab; ++q) {
      mbar_init(&S.full_a[q], CVT_WARPS);
      mbar_init(&S.empty_a[q], 1);
    }
    for (uint32_t q = 0; q < nring; ++q) {
      mbar_init(&S.full_b[q], 1);
      mbar_init(&S.empty_b[q], 1);
    }
    for (int b = 0; b < ACCS; ++b) {
      mbar_init(&S.nx_free[b], EPI_WARPS);
      mbar_init(&S.full_acc[b], 1);
      mbar_init(&S.empty_acc[b], EPI_WARPS);
      mbar_init(&S.xfull[b], EPI_WARPS);
      mbar_init(&S.xfree[b], FIN_WARPS);
    }
    mbar_init(&S.drained, 1);
    fence_mbar_init();
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&S.tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // everything read from here on was written by earlier kernels of the job
  pdl_wait();
  // columns without a centroid get an infinite norm, so they never win
  for (uint32_t t = threadIdx.x; t < nc * NMAX; t += WD_THREADS) cn[t] = t < k ? cnorm[t] : INFINITY;
  for (uint32_t t = threadIdx.x; t < DC_MAX_W * KD; t += WD_THREADS) S.center[t] = t < d ? center[t] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;
  const float cmax = __uint_as_float(*cmax_bits);

  if (warp >= CVT_WARP0 && warp < CVT_WARP0 + CVT_WARPS) {
    // ---------------------------------------------------------- converters
    // Warp cw owns tile rows 16 cw .., step q gives lane l row 16 cw + 2q +
    // l / 16 and dims 4 (l % 16) .. + 3 of each dimension chunk: one warp load
    // reads 256 contiguous bytes of two rows, one warp store writes two whole
    // 128-byte swizzled BF16 rows.
    const int r0 = (warp - CVT_WARP0) * CVT_ROWS, col = lane & 15, rsub = lane >> 4;
    const bool vec = d % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    unsigned int mabs = 0;  // bits of max |x|
    for (uint32_t i = 0;; ++i) {
      const uint32_t tile = blockIdx.x + i * gridDim.x;
      if (tile >= ntiles) break;
      const uint32_t ab = i % nab;
      uint8_t* A = base + ab * dc * 2 * A_TILE;
      float ss[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) ss[q] = 0.f;
      bool ok = true;
      for (uint32_t e = 0; e < dc; ++e) {
        const uint32_t d0 = e * KD + 4 * col;
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const uint32_t p = tile * TM + r0 + 2 * q + rsub;
          const float* row = x + (uint64_t)p * d + d0;
          v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (p < n && d0 < d) {
            if (vec) {
              v[q] = __ldg(reinterpret_cast<const float4*>(row));
            } else {
              v[q].x = __ldg(row);
              if (d0 + 1 < d) v[q].y = __ldg(row + 1);
              if (d0 + 2 < d) v[q].z = __ldg(row + 2);
              if (d0 + 3 < d) v[q].w = __ldg(row + 3);
            }
          }
        }
        if (e == 0) {
          if (i >= nab) ok = mbar_wait(&S.empty_a[ab], ((i / nab) + 1) & 1, err, polls);
          if (i >= 2) ok = ok && mbar_wait(&S.nx_free[i & 1], ((i / 2) + 1) & 1, err, polls);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        const float4 m = *reinterpret_cast<const float4*>(S.center + d0);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int rr = r0 + 2 * q + rsub;
          if (maxabs)
            mabs = max(mabs, max(max(__float_as_uint(fabsf(v[q].x)), __float_as_uint(fabsf(v[q].y))),
                                 max(__float_as_uint(fabsf(v[q].z)), __float_as_uint(fabsf(v[q].w)))));
          const float a0 = __fsub_rn(v[q].x, m.x), a1 = __fsub_rn(v[q].y, m.y);
          const float a2 = __fsub_rn(v[q].z, m.z), a3 = __fsub_rn(v[q].w, m.w);
          ss[q] = fmaf(a3, a3, fmaf(a2, a2, fmaf(a1, a1, fmaf(a0, a0, ss[q]))));
          uint32_t hi0, lo0, hi1, lo1;
          split2(a0, a1, hi0, lo0);
          split2(a2, a3, hi1, lo1);
          const uint32_t off = swz(rr, col >> 1) + (uint32_t)(col & 1) * 8u;
          *reinterpret_cast<uint2*>(A + e * 2 * A_TILE + off) = make_uint2(hi0, hi1);
          *reinterpret_cast<uint2*>(A + e * 2 * A_TILE + A_TILE + off) = make_uint2(lo0, lo1);
        }
      }
      if (!ok) break;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float s = ss[q];
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (col == 0) S.nx[i & 1][r0 + 2 * q + rsub] = s;
      }
      fence_proxy_async();  // the MMAs read the operands through the async proxy
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.full_a[ab]);
    }
    if (maxabs) {
      for (int o = 16; o; o >>= 1) mabs = max(mabs, __shfl_xor_sync(0xffffffffu, mabs, o));
      if (lane == 0) atomicMax(maxabs, mabs);
    }
  } else if (warp == COPY_WARP) {
    // -------------------------------------------- centroid operand producer
    if (lane == 0) {
      uint32_t u = 0;  // copies issued
      bool ok = true;
      for (uint32_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
        for (uint32_t ch = 0; ok && ch < nc; ++ch) {
          const uint32_t bytes = min((uint32_t)NMAX, npad - ch * NMAX) * 128;
          for (uint32_t e = 0; e < 2 * dc; ++e) {
            const uint32_t q = u % nring;
            if (u >= nring && !mbar_wait(&S.empty_b[q], ((u / nring) + 1) & 1, err, polls)) {
              ok = false;
              break;
            }
            mbar_expect_tx(&S.full_b[q], bytes);
            bulk_g2s(ring_b + q * OP_TILE, bop + (uint64_t)(ch * 2 * dc + e) * OP_TILE, bytes, &S.full_b[q]);
            ++u;
          }
        }
      }
      // No copy may still be landing when the CTA exits.  Copy u was issued
      // only after the MMAs that read copy u - nring had completed, so only
      // the last nring can be in flight.
      for (uint32_t i = u > nring ? u - nring : 0; i < u; ++i) mbar_drain(&S.full_b[i % nring], (i / nring) & 1);
    }
    __syncwarp();
  } else if (warp == MMA_WARP) {
    // ------------------------------------------------------------ MMA issue
    if (lane == 0) {
      uint32_t u = 0, cc = 0;  // centroid tiles and accumulators used so far
      bool ok = true;
      for (uint32_t i = 0; ok; ++i) {
        const uint32_t tile = blockIdx.x + i * gridDim.x;
        if (tile >= ntiles) break;
        const uint32_t ab = i % nab;
        if (!mbar_wait(&S.full_a[ab], (i / nab) & 1, err, polls)) break;
        const uint32_t A = su32(base + ab * dc * 2 * A_TILE);
        for (uint32_t ch = 0; ch < nc; ++ch, ++cc) {
          const uint32_t b = cc & 1, idesc = mma_idesc(min((uint32_t)NMAX, npad - ch * NMAX));
          if (cc >= (uint32_t)ACCS && !mbar_wait(&S.empty_acc[b], ((cc >> 1) + 1) & 1, err, polls)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dt = tmem + b * 256u;
          for (uint32_t e = 0; ok && e < dc; ++e) {
            const uint32_t ah = A + e * 2 * A_TILE, al = ah + A_TILE;
            for (int h = 0; h < 2; ++h, ++u) {
              const uint32_t q = u % nring;
              if (!mbar_wait(&S.full_b[q], (u / nring) & 1, err, polls)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t B = su32(ring_b + q * OP_TILE);
#pragma unroll
              for (int kk = 0; kk < KD / 16; ++kk) {
                const uint32_t o = kk * 32;
                mma_bf16(dt, sw128_desc(ah + o), sw128_desc(B + o), idesc, (e | h | kk) ? 1u : 0u);
                if (h == 0) mma_bf16(dt, sw128_desc(al + o), sw128_desc(B + o), idesc, 1u);
              }
              mma_commit(&S.empty_b[q]);
            }
          }
          if (!ok) break;
          mma_commit(&S.full_acc[b]);
        }
        if (ok) mma_commit(&S.empty_a[ab]);
      }
      // No MMA may still be running when TMEM is released or the operands go
      // away with the CTA: the commit arrives once every MMA issued above has
      // completed, waited for even when a wait gave up elsewhere.
      mma_commit(&S.drained);
      mbar_drain(&S.drained, 0);
    }
    __syncwarp();
  } else if (warp >= FIN_WARP0 && warp < FIN_WARP0 + FIN_WARPS) {
    // ------------------------------------------------------------ finalizers
    const int fw = warp - FIN_WARP0;
    const float eps_sum = 3.05f * 1.52587890625e-05f + (float)(3 * KD * dc + 8) * 2.384185791015625e-07f;
    const float eps32 = 1.01f * (float)(d + 12) * 5.9604644775390625e-08f;
    uint32_t moved = 0;  // this lane's points that changed cluster
    uint32_t cc = 0;
    bool ok = true;
    for (uint32_t tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x) {
      int t[FIN_QUADS][KM_CAND_MAX], rest[FIN_QUADS];
      uint32_t c[FIN_QUADS][KM_CAND_MAX], was[FIN_QUADS];
      float nxv[FIN_QUADS];
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        const uint32_t p = tile * TM + (uint32_t)((fw * FIN_QUADS + h) * 32 + lane);
        was[h] = nchg && p < n ? assign[p] & 0xffffu : 0u;
        rest[h] = KEY_NONE;
        nxv[h] = 0.f;
#pragma unroll
        for (uint32_t j = 0; j < KM_CAND_MAX; ++j) t[h][j] = KEY_NONE, c[h][j] = 0;
      }
      for (uint32_t ch = 0; ch < nc; ++ch, ++cc) {
        const uint32_t b = cc & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&S.xfull[b], (cc >> 1) & 1, err, polls));
        if (!ok) break;
#pragma unroll
        for (int h = 0; h < FIN_QUADS; ++h) {
          const int r = (fw * FIN_QUADS + h) * 32 + lane;
          nxv[h] = S.xnx[b][r];
#pragma unroll
          for (int u = 0; u < QUARTERS; ++u) {
            list_insert(t[h], c[h], rest[h], (int)S.xw1[b][u][r], ch * QUARTERS + u);
            list_insert(t[h], c[h], rest[h], (int)S.xw2[b][u][r], ch * QUARTERS + u);
            rest[h] = min(rest[h], (int)S.xlb[b][u][r]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.xfree[b]);
      }
      if (!ok) break;
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        const uint32_t p = tile * TM + (uint32_t)((fw * FIN_QUADS + h) * 32 + lane);
        bool flag = false, some = false;
        uint64_t cand = 0;
        uint32_t ncand = 0;
        if (p < n) {
          const float d1 = key_dist(t[h][0]), d2 = key_dist(t[h][1]);
          const float xn = sqrtf(nxv[h]);
          const float e = 2.f * eps_sum * xn * cmax + eps32 * (xn + cmax) * (xn + cmax) + 1e-36f;
          const float gap = 2.f * e + 6.103515625e-05f * d1;
          const float lim = fmaxf(1e-3f * d1, gap);
          if (t[h][0] < 0 || !(gap < INFINITY)) {
            flag = true;  // a negative smallest distance, or no bound at all: re-check
          } else if (d2 - d1 > lim) {
            const uint32_t now = c[h][0] / QUARTERS * NMAX + ((uint32_t)t[h][0] & 0xFFu);
            const uint32_t old = nchg ? was[h] : now;
            assign[p] = km_word(now, old);
            moved += now != old;
          } else {
#pragma unroll
            for (uint32_t j = 0; j < KM_CAND_MAX; ++j)
              if (key_dist(t[h][j]) - d1 <= lim) {
                const uint32_t cj = (uint32_t)t[h][j] & 0xFFu, first = c[h][j] / QUARTERS * NMAX;
                cand = (cand << 12) | (first + cj);
                ++ncand;
                // with another of its quarter's: what may hide behind both
#pragma unroll
                for (uint32_t i = 0; i < j; ++i)
                  if (c[h][i] == c[h][j]) {
                    const uint32_t c_lo = c[h][j] % QUARTERS * quarter_cols(min((uint32_t)NMAX, npad - first));
                    uint32_t h1, h2;
                    if (hidden_cols((uint32_t)t[h][i] & 0xFFu, cj, c_lo, h1, h2)) {
                      if (first + h1 < k) cand = (cand << 12) | (first + h1), ++ncand;
                      if (first + h2 < k) cand = (cand << 12) | (first + h2), ++ncand;
                    }
                  }
              }
            some = ncand >= 2 && ncand <= KM_CAND_MAX && key_dist(rest[h]) - d1 > gap;
            flag = !some;
          }
        }
        warp_append(some, nfew, lane, [&](uint32_t at) { few[at] = km_few(p, cand, ncand); });
        warp_append(flag, nlist, lane, [&](uint32_t at) { list[at] = p; });
      }
    }
    moved = __reduce_add_sync(0xffffffffu, moved);
    if (lane == 0 && moved) atomicAdd(nchg, moved);
  } else {
    // ------------------------------------------------------------- epilogue
    // Warp e reads TMEM lane quadrant e % 4 and column quarter e / 4 of each
    // accumulator, as in k_kmeans_tc.cu.
    const int q = warp & 3, quarter = warp >> 2;
    const int r = q * 32 + lane;
    uint32_t cc = 0;
    bool ok = true;
    for (uint32_t i = 0; ok; ++i) {
      const uint32_t tile = blockIdx.x + i * gridDim.x;
      if (tile >= ntiles) break;
      float nxv = 0.f;
      for (uint32_t ch = 0; ch < nc; ++ch, ++cc) {
        const uint32_t b = cc & 1, v = cc >> 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&S.full_acc[b], v & 1, err, polls));
        if (!ok) break;
        tc_fence_after();
        if (ch == 0) {
          nxv = S.nx[i & 1][r];
          __syncwarp();
          if (lane == 0) mbar_arrive(&S.nx_free[i & 1]);
        }
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + b * 256u;
        const uint32_t cols = min((uint32_t)NMAX, npad - ch * NMAX), cpq = quarter_cols(cols);
        const uint32_t c_lo = (uint32_t)quarter * cpq;
        int w1 = KEY_NONE, w2 = KEY_NONE, lb = KEY_NONE, col[GRID], row[GRID];
        if (c_lo < cols)
          quarter_keys(ta + c_lo, min(cpq, cols - c_lo), nxv, cn + ch * NMAX + c_lo, col, row,
                       SUMS ? sums + (((uint64_t)tile * TM + r) * nc + ch) * NMAX + c_lo : nullptr);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.empty_acc[b]);
        if (c_lo < cols) top2_grid(col, row, c_lo, w1, w2, lb);
        if (cc >= (uint32_t)ACCS) {
          ok = __all_sync(0xffffffffu, mbar_wait(&S.xfree[b], (v + 1) & 1, err, polls));
          if (!ok) break;
        }
        S.xw1[b][quarter][r] = (uint32_t)w1;
        S.xw2[b][quarter][r] = (uint32_t)w2;
        S.xlb[b][quarter][r] = (uint32_t)lb;
        if (quarter == 0) S.xnx[b][r] = nxv;
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.xfull[b]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0 && S.err) atomicAdd(timeouts, 1ull);
}

}  // namespace

bool km_wide_supported(uint32_t d, uint32_t k) { return d >= 1 && d <= DC_MAX_W * KD && k >= 1 && k <= K_MAX_W; }

size_t km_wide_operand_bytes(uint32_t d, uint32_t k) {
  return (size_t)cent_chunks(k) * dim_chunks(d) * 2 * OP_TILE;
}

cudaError_t launch_kmeans_wide_assign(const float* x, uint32_t n, uint32_t d, uint32_t k, KmBuffers& b,
                                      const unsigned int* cmax, uint32_t* nchg, const DevInfo& di, cudaStream_t s,
                                      uint64_t* nk, bool maxabs) {
  const uint32_t ntiles = (n + TM - 1) / TM;
  uint32_t grid = ntiles < (uint32_t)di.sms ? ntiles : (uint32_t)di.sms;
  if (b.grid_cap && grid > b.grid_cap) grid = b.grid_cap;
  const size_t smem = wide_smem(k);
  cudaError_t e = allow_smem<km_wide_assign_kernel<>>(di);
  if (e != cudaSuccess || (e = kt_begin(b.kt, s)) != cudaSuccess) return e;
  e = launch_pdl(km_wide_assign_kernel<>, dim3(grid), dim3(WD_THREADS), smem, s, x, n, d, k, (const uint8_t*)b.bop,
                 (const float*)b.center, (const float*)b.cnorm, cmax, b.assign, nchg, b.flagged, b.nflag + 1, b.pairs,
                 b.nflag + 4, b.stats + 3, (float*)nullptr, b.polls < 0 ? SPIN_LIMIT : b.polls,
                 maxabs ? b.maxabs : (unsigned int*)nullptr);
  if (e != cudaSuccess || (e = kt_end(b.kt, s)) != cudaSuccess) return e;
  ++*nk;
  return cudaSuccess;
}

}  // namespace mrgb
