// k-means assignment on the 5th-generation tensor cores (tcgen05): the
// points x centroids contraction in BF16 with FP32 accumulation in tensor
// memory (TMEM), followed by an exact re-check of near ties.
//
// The distance d(x, c) = ||x||^2 - 2 x.c + ||c||^2 needs the cross term x.c,
// a dense (points x D) . (D x K) contraction — the one step of the hot path
// that is a real GEMM.  Per tile of 128 points:
//   * for D = 64 one producer thread moves each FP32 tile (128 rows, 32 KB,
//     contiguous) into a two-deep shared-memory ring with one bulk copy
//     (cp.async.bulk, completion counted on an mbarrier), so loads stay in
//     flight without registers; 8 converter warps read the tile (rows
//     of the filter's list they fetch themselves, by 16-byte asynchronous copies a
//     tile ahead; for other D they load the values as they need them), compute ||x||^2 in FP32, and write BF16
//     operands in the 128-byte-swizzled K-major layout the MMA reads.  With TERMS = 3 each value is split as
//     x = hi + lo (hi = bf16(x), lo = bf16(x - hi)) and the MMA accumulates
//     hi.hi + hi.lo + lo.hi, so the cross term is good to about 2^-15
//     relative; TERMS = 1 is the plain single BF16 product.
//   * one thread issues tcgen05.mma (M = 128, N = K rounded up to 16, K = 16
//     per instruction, 4 steps over D = 64) into one of two 256-column TMEM
//     accumulators, and commits completion to mbarriers;
//   * 16 epilogue warps read the 128 x N FP32 tile with tcgen05.ld (one
//     TMEM lane per point; four warps per lane quadrant, each on a quarter
//     of the columns), form d~ = fma(-2, acc, ||x||^2) + ||c||^2, pack it
//     with its column into one sortable 32-bit key, and reduce the keys to the
//     minima of the rows and columns of a grid (quarter_keys), which hold the
//     two smallest keys plus a lower bound of the others, and hand them to
//   * 4 finalizer warps (one lane quadrant each), which merge the four
//     column quarters of each point and apply the margin tests below, so
//     that no epilogue warp carries the per-point tail on its own path.
//     (Per tile a finalizer waits for one list reservation and writes scattered
//     words and bounds; with two warps, two quadrants each, they set the pace:
//     the pass over 3.3M of 4M listed points took 977 us, with four 515.)
// Copies, converters, MMA issue, epilogue and finalizers overlap through the
// staging ring, two operand stages, two TMEM accumulators and two hand-off
// buffers.  Every mbarrier wait is bounded; on timeout the
// CTA stops, drains its MMAs, frees TMEM and reports through stats[3].
//
// Margin test (rigorous, per point).  With u_b = 2^-8 (BF16 rounding) the
// split leaves |x.c - (hi.hi + hi.lo + lo.hi)| <= 3.05 * 2^-16 ||x|| ||c||
// (one value: |x - hi - lo| <= u_b^2 |x|; sums by Cauchy-Schwarz); a single
// BF16 product leaves (2 u_b + u_b^2) ||x|| ||c||.  The tensor-core sum of the
// exact BF16 products is charged (products + 8) * 2^-22 ||x|| ||c|| (four
// times the round-to-nearest bound, allowing truncating adders; how the tensor
// core rounds is not documented, and the largest error that random and adverse
// operands show, 192 to 768 products, is 0.05 of the charge:
// tests/test_gpu_km_sums.py), and the FP32
// norms and the final fma/add (D + 8) * 2^-24 (||x|| + ||c||)^2 (Higham,
// eq. 3.5).  Points and centroids are first shifted by the mean m of the
// initial centroids, x' = fl(x - m) and c' = fl(c - m): distances do not
// change, but the bounds then scale with the spread of the data, not with
// its offset from zero.  Each subtraction is correctly rounded, so x' - c'
// differs from x - c by at most 2^-24 (||x'|| + ||c'||) and its square by at
// most twice that times (||x'|| + ||c'||): (D + 12) in place of (D + 8)
// covers it, and x, c stand for x', c' in all of the bounds here.  The keys hold d~ truncated to 16 mantissa bits (t <= d~ <
// t (1 + 2^-15)), so with G = 2E + 2^-14 t_1: if t_2 - t_1 > max(1e-3 t_1, G)
// the tensor-core winner is the exact winner.  Otherwise, if b > t_1 + G for a
// lower bound b of every key but each column quarter's two smallest, every
// centroid not among those with a key up to t_1 + max(1e-3 t_1, G) has exact
// distance above t_1 (1 + 2^-15) + E >= d(k_1); with at most KM_CAND_MAX of
// them the point needs an exact choice between those few alone, else it is
// listed and compared with every centroid (km_settle_kernel either way), so
// assignments equal the FP64 argmin.  (Two keys may hide behind a quarter's two
// smallest in its grid: they are above both, so they matter only when both are
// candidates, and then count as candidates too.)  A centroid that is not finite,
// or whose norm overflows, makes max ||c|| and with it E infinite or NaN: no
// test then holds, and every point is listed.
#include <type_traits>

#include "dev_tc.cuh"

namespace mrgb {
namespace {

using namespace tc;

constexpr int EPI_WARPS = 16;     // four per TMEM lane quadrant, each on a quarter of the columns
static_assert(EPI_WARPS == 4 * QUARTERS, "one warp per TMEM lane quadrant and column quarter");
constexpr int MMA_WARP = EPI_WARPS;
constexpr int CVT_WARP0 = MMA_WARP + 1;
constexpr int CVT_WARPS = 8;      // each converts TM / CVT_WARPS rows of a tile
constexpr int CVT_ROWS = TM / CVT_WARPS;
constexpr int FIN_WARP0 = CVT_WARP0 + CVT_WARPS;
constexpr int FIN_WARPS = 4;      // each finalizes 4 / FIN_WARPS TMEM lane quadrants (32 points each)
constexpr int FIN_QUADS = 4 / FIN_WARPS;
constexpr int TMA_WARP = FIN_WARP0 + FIN_WARPS;  // 29
constexpr int TC_THREADS = (EPI_WARPS + 1 + CVT_WARPS + FIN_WARPS + 1) * 32;  // 960
static_assert(CVT_ROWS % 16 == 0 && 4 % FIN_WARPS == 0, "converter rows and finalizer quadrants");
constexpr int STAGES = 2;         // operand stages
constexpr int XST = 2;            // FP32 staging buffers filled by the bulk copy engine
constexpr uint32_t BEYOND = 0xFFFFFFFFu;  // no point (n < 2^31)
constexpr uint32_t LISTED = 0xFFu;        // (number of candidates) too many: every centroid
constexpr int ACCS = 2;           // TMEM accumulators
constexpr uint32_t TMEM_COLS = 512;  // two 256-column FP32 accumulators
struct __align__(1024) TcSmem {
  uint8_t b_hi[NMAX * 128];
  uint8_t b_lo[NMAX * 128];
  uint8_t a_hi[STAGES][TM * 128];
  uint8_t a_lo[STAGES][TM * 128];
  float xs[XST][TM * KD];             // FP32 point tiles (D == 64 path)
  float nx[STAGES][TM];
  float cn[NMAX];
  float drift[NMAX];                  // (bounds) the centroids' drifts so far
  // per column quarter and row: top-2 keys and the lower bound of the
  // other keys; and the row's ||x||^2 (epilogue -> finalizers)
  uint32_t xw1[ACCS][QUARTERS][TM], xw2[ACCS][QUARTERS][TM], xlb[ACCS][QUARTERS][TM];
  float xnx[ACCS][TM];
  unsigned long long full_a[STAGES], empty_a[STAGES], nx_free[STAGES];
  unsigned long long full_acc[ACCS], empty_acc[ACCS], drained;
  unsigned long long xfull[ACCS], xfree[ACCS];  // epilogue warps hand their keys to the finalizers
  unsigned long long tfull[XST], tempty[XST];   // FP32 staging ring
  uint32_t tmem_base;
  int err;
};

static_assert(sizeof(TcSmem) + 1024 <= 232448, "shared memory of one CTA");

// a load that stays where it is written (its value is used a tile later)
__device__ __forceinline__ uint32_t ld_now(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// SUMS: the tensor core's sums of every point and column go to sums [tiles TM][NMAX]
// (tests/km_tc_sums.cu measures their error against the charge above).
template <int TERMS, bool SUMS = false>
__global__ void __launch_bounds__(TC_THREADS, 1)
km_tc_assign_kernel(const float* __restrict__ x, uint32_t n_all, uint32_t d, const float* __restrict__ c, uint32_t k,
                    const float* __restrict__ center, const float* __restrict__ cnorm, const unsigned int* cmax_bits, uint32_t* __restrict__ assign, uint32_t* nchg,
                    uint32_t* __restrict__ list, uint32_t* nlist, KmFew* __restrict__ pairs, uint32_t* npairs,
                    unsigned long long* timeouts, float* sums, long long polls, uint32_t stop_copies,
                    unsigned int* maxabs, const uint32_t* __restrict__ act, const uint32_t* nact, KmBounds B) {
  extern __shared__ uint8_t tc_raw[];
  TcSmem& S = *reinterpret_cast<TcSmem*>((reinterpret_cast<uintptr_t>(tc_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t npad = (k + 15) & ~15u;
  volatile int* err = &S.err;

  if (threadIdx.x == 0) {
    S.err = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&S.full_a[s], CVT_WARPS);
      mbar_init(&S.empty_a[s], 1);
      mbar_init(&S.nx_free[s], EPI_WARPS);
    }
    for (int b = 0; b < ACCS; ++b) {
      mbar_init(&S.full_acc[b], 1);
      mbar_init(&S.empty_acc[b], EPI_WARPS);
      mbar_init(&S.xfull[b], EPI_WARPS);
      mbar_init(&S.xfree[b], FIN_WARPS);
    }
    for (int q = 0; q < XST; ++q) mbar_init(&S.tempty[q], CVT_WARPS);
    mbar_init(&S.drained, 1);
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&S.tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // everything read from here on was written by earlier kernels of the job
  pdl_wait();
  // the points: all of them, or those the filter listed (unless that is nearly all)
  const uint32_t* idx = act && km_use_list(*nact, n_all) ? act : nullptr;
  const uint32_t n = idx ? *nact : n_all;
  const uint32_t ntiles = (n + TM - 1) / TM;
  if (threadIdx.x == 0) {
    for (int q = 0; q < XST; ++q) mbar_init(&S.tfull[q], 1);
    fence_mbar_init();
  }
  // Points of KD aligned values are staged in shared memory: whole tiles by the
  // copy engine, the rows of the filter's list by the converters.
  const bool vec = d == KD && ((reinterpret_cast<uintptr_t>(x) & 15) == 0);
  const bool gather = vec && idx, bulk = vec && !idx;
  // The dimension in column p of the operands.  Other points than those keep
  // dimensions 16 apart in a lane's four columns (the contraction does not
  // mind): a warp's load then reads 64 contiguous bytes of two rows, and there
  // are only as many loads as D needs (800,000 x 37, K = 100, ten rounds 1.152 ->
  // 1.132 ms).
  auto dim_at = [&](uint32_t p) { return vec ? p : (p >> 2) + 16 * (p & 3); };
  // centroid operands (rows >= k and dims >= d are zero) and norms
  for (uint32_t t = threadIdx.x; t < npad * (KD / 2); t += blockDim.x) {
    const uint32_t row = t / (KD / 2), pr = t % (KD / 2);
    const uint32_t d0 = dim_at(2 * pr), d1 = dim_at(2 * pr + 1);
    float a = 0.f, b = 0.f;
    if (row < k) {
      if (d0 < d) a = __fsub_rn(c[(uint64_t)row * d + d0], center[d0]);
      if (d1 < d) b = __fsub_rn(c[(uint64_t)row * d + d1], center[d1]);
    }
    uint32_t hi, lo;
    split2(a, b, hi, lo);
    const uint32_t off = swz((int)row, (int)(pr >> 2)) + (pr & 3) * 4;
    *reinterpret_cast<uint32_t*>(S.b_hi + off) = hi;
    *reinterpret_cast<uint32_t*>(S.b_lo + off) = lo;
  }
  // padded centroid columns get an infinite norm, so they never win
  for (uint32_t t = threadIdx.x; t < NMAX; t += blockDim.x) {
    S.cn[t] = t < k ? cnorm[t] : INFINITY;
    S.drift[t] = B.ub && t < k ? B.drift[t] : 0.f;
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem_base;
  const float cmax = __uint_as_float(*cmax_bits);

  if (warp >= CVT_WARP0 && warp < CVT_WARP0 + CVT_WARPS) {
    // ---------------------------------------------------------- converters
    // Warp cw owns tile rows CVT_ROWS cw .., in parts of 16.  Step q of part
    // hf gives lane l row CVT_ROWS cw + 16 hf + 2q + l / 16 and dims
    // 4 (l % 16) .. + 3, so one warp load reads two whole FP32 rows (512
    // contiguous bytes) and one warp store writes two whole 128-byte
    // swizzled BF16 rows: no shared-memory bank conflicts.
    const int cw = warp - CVT_WARP0;
    const int col = lane & 15, rsub = lane >> 4;
    float mv[4];  // the shift of this lane's four dimensions
#pragma unroll
    for (int j = 0; j < 4; ++j) mv[j] = dim_at(4 * col + j) < d ? center[dim_at(4 * col + j)] : 0.f;
    // Listed rows: each warp fetches its own rows of the next tile while it
    // converts this one, 16 bytes a lane and two rows per instruction, the row
    // numbers a tile ahead of that.  (By the copy warp, through the barriers of
    // the staging ring, each tile waited for the row numbers, the copies and a
    // hand-over in turn: 3.3M of 4M listed points 517 us, now 431; one bulk
    // copy per row 817.)
    const uint32_t r0w = CVT_ROWS * cw;
    auto list_row = [&](uint32_t t) {
      const uint32_t r = t * TM + r0w + lane;
      return t < ntiles && lane < CVT_ROWS && r < n ? ld_now(idx + r) : BEYOND;
    };
    auto fetch = [&](uint32_t listed, uint32_t slot) {  // lane r: row r
#pragma unroll
      for (int t = 0; t < CVT_ROWS / 2; ++t) {
        const uint32_t r = 2 * t + rsub, p = __shfl_sync(0xffffffffu, listed, r);
        if (p != BEYOND) cp_async16(&S.xs[slot][(r0w + r) * KD + 4 * col], x + (uint64_t)p * KD + 4 * col);
      }
      cp_async_commit();
    };
    static_assert(CVT_ROWS <= 32 && XST == 2, "a lane per row; two fetched tiles");
    unsigned int mabs = 0;  // bits of max |x| over the values this thread converts (non-negative floats order as ints)
    // (a loop of its own for listed rows: sharing one cost the other paths 5%)
    auto convert = [&](auto gather_t) {
      constexpr bool GATHER = decltype(gather_t)::value;
      uint32_t listed = 0;  // the rows of the tile fetched next
      if (GATHER) {
        fetch(list_row(blockIdx.x), 0);
        listed = list_row(blockIdx.x + gridDim.x);
      }
      for (uint32_t i = 0;; ++i) {
        const uint32_t tile = blockIdx.x + i * gridDim.x;
        if (tile >= ntiles) break;
        const int s = (int)(i % STAGES);
        const uint32_t u = i / STAGES;
        const int q2 = (int)(i % XST);
        if (!GATHER && vec) {
          // the tile was staged by the bulk copy engine
          const bool okt = mbar_wait(&S.tfull[q2], (i / XST) & 1, err, polls);
          if (!__all_sync(0xffffffffu, okt)) break;
        } else if (GATHER) {
          fetch(listed, (i + 1) & 1);
          listed = list_row(tile + 2 * gridDim.x);
          cp_async_wait<1>();
          __syncwarp();
        }
        bool ok = true;
        for (int hf = 0; hf < CVT_ROWS / 16; ++hf) {
          const int r0 = CVT_ROWS * cw + 16 * hf;
          float4 v[8];
          if (GATHER || vec) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int rr = r0 + 2 * q + rsub;
              v[q] = tile * TM + rr < n ? *reinterpret_cast<const float4*>(&S.xs[q2][rr * KD + 4 * col])
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const uint32_t p = tile * TM + r0 + 2 * q + rsub;
              const float* row = x + (uint64_t)(idx && p < n ? idx[p] : p) * d + col;
              const uint32_t left = p < n && (uint32_t)col < d ? d - col : 0;
              v[q].x = left > 0 ? row[0] : 0.f;
              v[q].y = left > 16 ? row[16] : 0.f;
              v[q].z = left > 32 ? row[32] : 0.f;
              v[q].w = left > 48 ? row[48] : 0.f;
            }
          }
          if (hf == 0 && i >= STAGES) {
            ok = mbar_wait(&S.empty_a[s], (u + 1) & 1, err, polls);
            ok = ok && mbar_wait(&S.nx_free[s], (u + 1) & 1, err, polls);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
          }
          float ss[8];  // this lane's part of its eight rows' norms
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int rr = r0 + 2 * q + rsub;
            if (maxabs)
              mabs = max(mabs, max(max(__float_as_uint(fabsf(v[q].x)), __float_as_uint(fabsf(v[q].y))),
                                   max(__float_as_uint(fabsf(v[q].z)), __float_as_uint(fabsf(v[q].w)))));
            v[q].x = __fsub_rn(v[q].x, mv[0]);
            v[q].y = __fsub_rn(v[q].y, mv[1]);
            v[q].z = __fsub_rn(v[q].z, mv[2]);
            v[q].w = __fsub_rn(v[q].w, mv[3]);
            ss[q] = fmaf(v[q].w, v[q].w, fmaf(v[q].z, v[q].z, fmaf(v[q].y, v[q].y, v[q].x * v[q].x)));
            uint32_t hi0, lo0, hi1, lo1;
            split2(v[q].x, v[q].y, hi0, lo0);
            split2(v[q].z, v[q].w, hi1, lo1);
            const uint32_t off = swz(rr, col >> 1) + (uint32_t)(col & 1) * 8u;
            *reinterpret_cast<uint2*>(S.a_hi[s] + off) = make_uint2(hi0, hi1);
            if (TERMS == 3) *reinterpret_cast<uint2*>(S.a_lo[s] + off) = make_uint2(lo0, lo1);
          }
          // the 16 lanes' sums of eight rows at once: half of the rows stay at
          // each exchange (8 shuffles in place of 32)
#pragma unroll
          for (int w = 4; w; w >>= 1) {
            const bool up = col & 2 * w;
#pragma unroll
            for (int q = 0; q < w; ++q)
              ss[q] = (up ? ss[q + w] : ss[q]) + __shfl_xor_sync(0xffffffffu, up ? ss[q] : ss[q + w], 2 * w);
          }
          ss[0] += __shfl_xor_sync(0xffffffffu, ss[0], 1);
          if ((col & 1) == 0) S.nx[s][r0 + 2 * (col >> 1) + rsub] = ss[0];
        }
        if (!ok) break;
        // The staging buffer is released only here: the bulk copy engine writes
        // through the async proxy, so the shared loads above must be ordered
        // before its next fill by this proxy fence (the stores that consumed
        // them precede it), not just by the mbarrier arrive.
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&S.full_a[s]);
          if (!GATHER && vec) mbar_arrive(&S.tempty[q2]);
        }
      }
      if (GATHER) cp_async_wait<0>();
    };
    if (gather) convert(std::true_type{});
    else convert(std::false_type{});
    if (maxabs) {
      for (int o = 16; o; o >>= 1) mabs = max(mabs, __shfl_xor_sync(0xffffffffu, mabs, o));
      if (lane == 0) atomicMax(maxabs, mabs);
    }
  } else if (warp == TMA_WARP) {
    // ------------------------------------------------- bulk-copy producer
    // one bulk copy per tile
    if (bulk && lane == 0) {
      uint32_t issued = 0;
      for (uint32_t i = 0;; ++i) {
        const uint32_t tile = blockIdx.x + i * gridDim.x;
        if (tile >= ntiles || (stop_copies && i >= stop_copies)) break;
        const int q2 = (int)(i % XST);
        const uint32_t rows = (n - tile * TM) < (uint32_t)TM ? (n - tile * TM) : (uint32_t)TM;
        if (i >= XST && !mbar_wait(&S.tempty[q2], ((i / XST) + 1) & 1, err, polls)) break;
        mbar_expect_tx(&S.tfull[q2], rows * KD * 4);
        bulk_g2s(S.xs[q2], x + (uint64_t)tile * TM * KD, rows * KD * 4, &S.tfull[q2]);
        ++issued;
      }
      // No copy may still be landing in shared memory when the CTA exits.
      // Copy i was issued only after the converters released copy i - XST
      // (which they do after its completion), so only the last XST copies
      // can be in flight; wait for them even when a wait gave up elsewhere.
      for (uint32_t i = issued > (uint32_t)XST ? issued - XST : 0; i < issued; ++i)
        mbar_drain(&S.tfull[i % XST], (i / XST) & 1);
    }
    __syncwarp();
  } else if (warp == MMA_WARP) {
    // ------------------------------------------------------------ MMA issue
    if (lane == 0) {
      const uint32_t idesc = mma_idesc(npad);
      const uint32_t bh = su32(S.b_hi), bl = su32(S.b_lo);
      uint32_t issued = 0;
      for (uint32_t i = 0;; ++i) {
        const uint32_t tile = blockIdx.x + i * gridDim.x;
        if (tile >= ntiles) break;
        const int s = (int)(i % STAGES);
        const uint32_t u = i / STAGES;
        const int b = (int)(i & 1);
        const uint32_t v = i >> 1;
        if (!mbar_wait(&S.full_a[s], u & 1, err, polls)) break;
        if (i >= ACCS && !mbar_wait(&S.empty_acc[b], (v + 1) & 1, err, polls)) break;
        tc_fence_after();
        const uint32_t dt = tmem + (uint32_t)b * 256u;
        const uint32_t ah = su32(S.a_hi[s]), al = su32(S.a_lo[s]);
#pragma unroll
        for (int kk = 0; kk < KD / 16; ++kk) {
          const uint32_t o = kk * 32;  // 16 BF16 = 32 bytes along K inside the swizzle row
          mma_bf16(dt, sw128_desc(ah + o), sw128_desc(bh + o), idesc, kk > 0 ? 1u : 0u);
          if (TERMS == 3) {
            mma_bf16(dt, sw128_desc(ah + o), sw128_desc(bl + o), idesc, 1u);
            mma_bf16(dt, sw128_desc(al + o), sw128_desc(bh + o), idesc, 1u);
          }
        }
        mma_commit(&S.empty_a[s]);
        mma_commit(&S.full_acc[b]);
        ++issued;
      }
      // No MMA may still be running when TMEM is released (or when the
      // operand buffers go away with the CTA): the commit arrives once every
      // MMA issued above has completed, and that is waited for even when a
      // wait gave up elsewhere.
      if (issued) {
        mma_commit(&S.drained);
        mbar_drain(&S.drained, 0);
      }
    }
    __syncwarp();
  } else if (warp >= FIN_WARP0 && warp < FIN_WARP0 + FIN_WARPS) {
    // ------------------------------------------------------------ finalizers
    // Warp f takes the points of TMEM lane quadrants FIN_QUADS f .. (rows
    // 32 q + lane of each): it merges the four column quarters' top-2 keys
    // into the row's exact top-2 (g1, g2), then applies the margin tests.
    const int fw = warp - FIN_WARP0;
    const float eps_sum = TERMS == 3 ? (3.05f * 1.52587890625e-05f + (float)(3 * KD + 8) * 2.384185791015625e-07f)
                                     : (2.f * 3.90625e-03f + 1.52587890625e-05f + (float)(KD + 8) * 2.384185791015625e-07f);
    const float eps32 = 1.01f * (float)(d + 12) * 5.9604644775390625e-08f;
    uint32_t moved = 0;  // this lane's points that changed cluster
    const bool bounds = km_keeps_bounds(B);
    const float far = bounds ? *B.far : 0.f;
    // the points of the next two tiles and the words of the next one, so that no
    // load waits for another
    uint32_t p[FIN_QUADS], word[FIN_QUADS], p1[FIN_QUADS], word1[FIN_QUADS], p2[FIN_QUADS];
    auto load_points = [&](uint32_t tile, uint32_t (&to)[FIN_QUADS]) {
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        const uint32_t r = tile * TM + (uint32_t)((fw * FIN_QUADS + h) * 32 + lane);
        to[h] = tile >= ntiles || r >= n ? BEYOND : idx ? idx[r] : r;
      }
    };
    auto load_words = [&](const uint32_t (&of)[FIN_QUADS], uint32_t (&to)[FIN_QUADS]) {
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) to[h] = nchg && of[h] != BEYOND ? assign[of[h]] : 0u;
    };
    load_points(blockIdx.x, p1);
    load_points(blockIdx.x + gridDim.x, p2);
    load_words(p1, word1);
    for (uint32_t i = 0;; ++i) {
      const uint32_t tile = blockIdx.x + i * gridDim.x;
      if (tile >= ntiles) break;
      const int b = (int)(i & 1);
      const uint32_t v = i >> 1;
      const bool okx = mbar_wait(&S.xfull[b], v & 1, err, polls);
      if (!__all_sync(0xffffffffu, okx)) break;
      int o1[FIN_QUADS][QUARTERS], o2[FIN_QUADS][QUARTERS], ol[FIN_QUADS][QUARTERS];
      float nxv[FIN_QUADS];
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        const int r = (fw * FIN_QUADS + h) * 32 + lane;
#pragma unroll
        for (int u = 0; u < QUARTERS; ++u) {
          o1[h][u] = (int)S.xw1[b][u][r];
          o2[h][u] = (int)S.xw2[b][u][r];
          ol[h][u] = (int)S.xlb[b][u][r];
        }
        nxv[h] = S.xnx[b][r];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.xfree[b]);
      uint32_t ncand[FIN_QUADS];
      uint64_t cand[FIN_QUADS];
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) p[h] = p1[h], word[h] = word1[h], p1[h] = p2[h];
      load_words(p1, word1);
      load_points(tile + 2 * gridDim.x, p2);
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        int g1 = o1[h][0], g2 = o2[h][0];
#pragma unroll
        for (int u = 1; u < QUARTERS; ++u) top2_merge(g1, g2, o1[h][u], o2[h][u]);
        cand[h] = 0;
        ncand[h] = 0;  // 0: decided; 2 .. KM_CAND_MAX: few; LISTED
        if (p[h] != BEYOND) {
          const float d1 = key_dist(g1), d2 = key_dist(g2);
          const float xn = km_sqrt(nxv[h]) * 1.000001f;
          // (1e-36: the products of tiny values may be flushed to zero)
          const float e = 2.f * eps_sum * xn * cmax + eps32 * (xn + cmax) * (xn + cmax) + 1e-36f;
          // keys under-state a distance by less than 2^-15 of it (2^-14 allowed)
          const float gap = 2.f * e + 6.103515625e-05f * d1;
          const float lim = fmaxf(1e-3f * d1, gap);
          if (g1 < 0 || !(gap < INFINITY)) {
            ncand[h] = LISTED;  // a negative smallest distance, or no bound at all: re-check
          } else if (d2 - d1 > lim) {
            const uint32_t now = (uint32_t)g1 & 0xFFu, o = nchg ? word[h] & 0xffffu : now;
            assign[p[h]] = km_word(now, o);
            moved += now != o;
            if (bounds) km_put_bounds(B, p[h], S.drift[now], far, fmaf(d1, 1.00006103515625f, e), d2 - e);
          } else {
            const uint32_t cpq = quarter_cols(npad);
            // candidates: the quarters' top-2 keys within the margin and what
            // may hide behind both of a quarter's, if every other key is beyond it
            int rest = KEY_NONE;
            uint32_t nc = 0;
#pragma unroll
            for (uint32_t u = 0; u < QUARTERS; ++u) {
              rest = min(rest, ol[h][u]);
              auto add = [&](uint32_t column) {
                cand[h] = (cand[h] << 12) | column;
                ++nc;
              };
              const uint32_t c1 = (uint32_t)o1[h][u] & 0xFFu, c2 = (uint32_t)o2[h][u] & 0xFFu;
              if (key_dist(o1[h][u]) - d1 <= lim) add(c1);
              else rest = min(rest, o1[h][u]);
              if (key_dist(o2[h][u]) - d1 <= lim) {
                add(c2);
                uint32_t h1, h2;
                if (hidden_cols(c1, c2, u * cpq, h1, h2)) {
                  if (h1 < k) add(h1);
                  if (h2 < k) add(h2);
                }
              } else {
                rest = min(rest, o2[h][u]);
              }
            }
            const bool few = key_dist(rest) - d1 > gap && nc >= 2 && nc <= KM_CAND_MAX;
            ncand[h] = few ? nc : LISTED;
            // (the settle pass lowers it by the candidates' distances)
            if (bounds && few) B.lb[p[h]] = km_sqrt(fmaxf(key_dist(rest) - e, 0.f)) * 0.999999f;
          }
        }
      }
      // one reservation in each list for all of the warp's points, both at once
      unsigned mf[FIN_QUADS], ml[FIN_QUADS];
      uint32_t tf = 0, tl = 0;
#pragma unroll
      for (int h = 0; h < FIN_QUADS; ++h) {
        mf[h] = __ballot_sync(0xffffffffu, ncand[h] != 0 && ncand[h] != LISTED);
        ml[h] = __ballot_sync(0xffffffffu, ncand[h] == LISTED);
        tf += __popc(mf[h]);
        tl += __popc(ml[h]);
      }
      if (tf + tl) {
        uint32_t base = 0;
        if (lane == 0 && tf) base = atomicAdd(npairs, tf);
        if (lane == 1 && tl) base = atomicAdd(nlist, tl);
        uint32_t bf = __shfl_sync(0xffffffffu, base, 0), bl = __shfl_sync(0xffffffffu, base, 1);
        const uint32_t below = (1u << lane) - 1;
#pragma unroll
        for (int h = 0; h < FIN_QUADS; ++h) {
          if (mf[h] >> lane & 1) pairs[bf + __popc(mf[h] & below)] = km_few(p[h], cand[h], ncand[h]);
          if (ml[h] >> lane & 1) list[bl + __popc(ml[h] & below)] = p[h];
          bf += __popc(mf[h]);
          bl += __popc(ml[h]);
        }
      }
    }
    moved = __reduce_add_sync(0xffffffffu, moved);
    if (lane == 0 && moved) atomicAdd(nchg, moved);
  } else {
    // ------------------------------------------------------------- epilogue
    // Warp e reads TMEM lane quadrant e % 4 (rows 32 (e % 4) ..) and column
    // quarter e / 4, CHUNK columns per tcgen05.ld.  Each distance becomes one
    // sortable 32-bit key (see dist_key); the keys are reduced to the minima of
    // the rows and columns of an 8 x 8 grid, those to the quarter's two smallest
    // (w1, w2) and a lower bound lb of the others, which go to the finalizer of
    // its lane quadrant.
    // (A running top-2, three minima and maxima per key, with the columns past K
    // masked one by one and up to 128 columns left to two of the quarters: 4M x
    // 64, K = 256, ten rounds 3.88 ms, now 3.70; 1M x 8, K = 20, one pass 112
    // us, now 108; 250,000 x 128, K = 512, five rounds 1.15 ms, now 1.12.)
    const int q = warp & 3, quarter = warp >> 2;
    const int r = q * 32 + lane;
    const uint32_t cols = npad, cpq = quarter_cols(cols), c_lo = (uint32_t)quarter * cpq;
    for (uint32_t i = 0;; ++i) {
      const uint32_t tile = blockIdx.x + i * gridDim.x;
      if (tile >= ntiles) break;
      const int s = (int)(i % STAGES);
      const int b = (int)(i & 1);
      const uint32_t v = i >> 1;
      const bool ok = mbar_wait(&S.full_acc[b], v & 1, err, polls);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const float nxv = S.nx[s][r];
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.nx_free[s]);
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * 256u;
      int w1 = KEY_NONE, w2 = KEY_NONE, lb = KEY_NONE, col[GRID], row[GRID];
      if (c_lo < cols)
        quarter_keys(ta + c_lo, min(cpq, cols - c_lo), nxv, S.cn + c_lo, col, row,
                     SUMS ? sums + ((uint64_t)tile * TM + r) * NMAX + c_lo : nullptr);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.empty_acc[b]);
      if (c_lo < cols) top2_grid(col, row, c_lo, w1, w2, lb);
      if (i >= ACCS) {
        const bool okf = mbar_wait(&S.xfree[b], (v + 1) & 1, err, polls);
        if (!__all_sync(0xffffffffu, okf)) break;
      }
      S.xw1[b][quarter][r] = (uint32_t)w1;
      S.xw2[b][quarter][r] = (uint32_t)w2;
      S.xlb[b][quarter][r] = (uint32_t)lb;
      if (quarter == 0) S.xnx[b][r] = nxv;
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.xfull[b]);
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

bool km_tc_supported(uint32_t d, uint32_t k) { return d >= 1 && d <= KD && k >= 1 && k <= NMAX; }

size_t km_tc_smem_bytes() { return sizeof(TcSmem) + 1024; }

// Raw launch: nchg (null in a job's first round, whose words hold nothing yet)
// counts the points that changed cluster; list/nlist receive the points to re-check, pairs/npairs the
// few-candidate points; act/nact (or null) name the points to take; maxabs (when not null) receives the bits of max |x|.
template <int TERMS, bool SUMS = false>
cudaError_t launch_km_tc_kernel(const float* x, uint32_t n, uint32_t d, const float* c, uint32_t k,
                                const float* center, const float* cnorm, const unsigned int* cmax_bits,
                                uint32_t* assign, uint32_t* nchg, uint32_t* list, uint32_t* nlist, KmFew* pairs,
                                uint32_t* npairs, unsigned long long* timeouts, float* sums, int grid, cudaStream_t s,
                                long long polls, uint32_t stop_copies, unsigned int* maxabs, const uint32_t* act,
                                const uint32_t* nact, const KmBounds& B) {
  const int smem = (int)km_tc_smem_bytes();
  const cudaError_t e = cudaFuncSetAttribute(km_tc_assign_kernel<TERMS, SUMS>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(km_tc_assign_kernel<TERMS, SUMS>, dim3(grid), dim3(TC_THREADS), (size_t)smem, s, x, n, d, c, k,
                    center, cnorm, cmax_bits, assign, nchg, list, nlist, pairs, npairs, timeouts, sums, polls,
                    stop_copies, maxabs, act, nact, B);
}

cudaError_t launch_kmeans_tc_assign(const float* x, uint32_t n, uint32_t d, const float* c, uint32_t k,
                                    KmBuffers& b, const unsigned int* cmax, uint32_t* nchg, const DevInfo& di,
                                    cudaStream_t s, uint64_t* nk, bool maxabs, const uint32_t* act,
                                    const uint32_t* nact) {
  const uint32_t ntiles = (n + TM - 1) / TM;
  uint32_t grid = ntiles < (uint32_t)di.sms ? ntiles : (uint32_t)di.sms;
  if (b.grid_cap && grid > b.grid_cap) grid = b.grid_cap;
  auto launch = b.precision == MR_KM_BF16X1_TC ? launch_km_tc_kernel<1> : launch_km_tc_kernel<3>;
  cudaError_t e = kt_begin(b.kt, s);
  if (e != cudaSuccess) return e;
  e = launch(x, n, d, c, k, b.center, b.cnorm, cmax, b.assign, nchg, b.flagged, b.nflag + 1, b.pairs, b.nflag + 4,
             b.stats + 3, nullptr, (int)grid, s, b.polls < 0 ? SPIN_LIMIT : b.polls, b.stop_copies,
             maxabs ? b.maxabs : nullptr, act, nact, b.bounds);
  if (e != cudaSuccess || (e = kt_end(b.kt, s)) != cudaSuccess) return e;
  ++*nk;
  // the caller re-checks the pairs and the listed near ties
  return cudaSuccess;
}

}  // namespace mrgb
