// k-means (Lloyd) as a MapReduce job with an array container.
//
// map (per point): key = index of the nearest centroid (squared Euclidean,
// lowest index on an exact tie), value = the point; combiner/reduce: per-key
// sum of points and count (K*D + K array); the new centroid is sum / count.
// The paper's array container with local arrays (Sec. III-A, III-E) is a
// per-CTA shared-memory copy of the K*D sums, merged into the global array.
//
// Exactness contract: assignments equal the FP64 argmin of
//   d(x, c) = sum_j ((double)x_j - (double)c_j)^2   (j in order, no FMA),
// and centroids are the exact-sum means rounded to FP32.
//
// A round is: the filter, in jobs where it pays (km_half_kernel,
// km_filter_kernel: points that provably keep their cluster are left out); the
// distance pass; the choice of what that left open (km_settle_kernel); the
// update of the sums; the next centroids (km_finalize_kernel).
//  * Distance pass: on the tensor cores for BF16 jobs and for FP32 jobs of up to
//    256 dimensions and 4,096 centroids (k_kmeans_tc.cu, k_kmeans_wide.cu, with
//    their bounds), else, and in contexts with a wait limit of their own, in
//    FP32 FMAs here (km_assign_fp32_kernel): d~ = ||x||^2 - 2 x.c + ||c||^2,
//    whose error is at most E = gamma_{D+3} (||x|| + ||c||)^2 (Higham, Accuracy
//    and Stability of Numerical Algorithms, eq. 3.4 / 3.5 for dot products); we
//    use E = 1.01 (D + 8) 2^-24 (||x|| + max_k ||c_k||)^2.  If the two smallest
//    d~ differ by more than 2E the FP32 winner is the FP64 winner.
//  * Every other point is settled by FP32 direct differences, whose relative
//    error is at most g = gamma_{D+3} (Higham, eq. 3.5 on a sum of squares), and
//    where those lie within (1 + g) / (1 - g) of each other by the definition in
//    FP64, with its order of operations.
//  * Sums are int64 fixed point, q = rint(x * 2^s), with s chosen from max|x| and
//    N so no sum can overflow; integer addition is exact and order-independent,
//    so results do not depend on scheduling.  A round in which few points moved
//    changes the sums by those alone; a full update adds runs of points of one
//    cluster in registers, after sorting windows of points by cluster in shared
//    memory (D <= 64) or all of them in global memory (K x D sums beyond one
//    CTA), or adds every coordinate in shared memory (the other shapes).
#include <cmath>

#include "dev_tc.cuh"

namespace mrgb {
namespace {

constexpr int KM_THREADS = 256;   // 8 warps
constexpr int TP = 64;            // points per tile (8 per warp)
constexpr int KC_MAX = 256;       // centroids per chunk (8 per lane)
constexpr int DC_MAX = 64;        // dims per chunk
constexpr int CS_LD = KC_MAX + 1;  // staged centroid row stride: the transposing stores hit distinct banks
constexpr int XS_LD = TP + 4;      // staged point row stride (16-byte rows; see the point loads)

// Running top three distances (the two smallest with their indices);
// between equal distances the lower index ranks first.
struct Top3 {
  float d1, d2, d3;
  int k1, k2;
};
__device__ __forceinline__ void top3_init(Top3& t) {
  t.d1 = t.d2 = t.d3 = INFINITY;
  t.k1 = t.k2 = 0x7fffffff;
}
__device__ __forceinline__ void top3_push(Top3& t, float d, int k) {
  if (d < t.d1 || (d == t.d1 && k < t.k1)) {
    t.d3 = t.d2;
    t.d2 = t.d1;
    t.k2 = t.k1;
    t.d1 = d;
    t.k1 = k;
  } else if (d < t.d2 || (d == t.d2 && k < t.k2)) {
    t.d3 = t.d2;
    t.d2 = d;
    t.k2 = k;
  } else if (d < t.d3) {
    t.d3 = d;
  }
}
// merge another triple in (its third index is never needed: a third value
// can only rank third)
__device__ __forceinline__ void top3_merge(Top3& t, const Top3& o) {
  top3_push(t, o.d1, o.k1);
  top3_push(t, o.d2, o.k2);
  top3_push(t, o.d3, 0x7fffffff);
}

// Sortable keys (K <= 256): the FP32 bits of a distance (negatives, which
// only rounding produces, clamped to 0) with the low 8 mantissa bits replaced
// by the centroid index.  Non-negative floats order like their bits, so keys
// order by the distance truncated to 16 mantissa bits (an under-statement of
// less than 2^-15 of it), then by index; a running top-2 is three unsigned
// min/max.  KEY_NONE (no centroid) decodes to +inf.
constexpr uint32_t KEY_NONE = 0x7F8000FFu;
__device__ __forceinline__ uint32_t dist_key(float dist, uint32_t kk) {
  return ((uint32_t)max((int)__float_as_uint(dist), 0) & 0xFFFFFF00u) | kk;
}
__device__ __forceinline__ float key_dist(uint32_t key) { return __uint_as_float(key & 0xFFFFFF00u); }
__device__ __forceinline__ void top2_insert(uint32_t& t1, uint32_t& t2, uint32_t key) {
  const uint32_t h = max(t1, key);
  t1 = min(t1, key);
  t2 = min(t2, h);
}
// (a1 <= a2, every other key of set a >= la) merged with the same of set b:
// the union's top-2 and a lower bound of its other keys.
__device__ __forceinline__ void top2lb_merge(uint32_t& a1, uint32_t& a2, uint32_t& la, uint32_t b1, uint32_t b2,
                                             uint32_t lb) {
  const uint32_t g1 = min(a1, b1);
  const uint32_t g2 = min(max(a1, b1), min(a2, b2));
  uint32_t g3 = min(la, lb);
  g3 = (a1 != g1 && a1 != g2) ? min(g3, a1) : g3;
  g3 = (a2 != g1 && a2 != g2) ? min(g3, a2) : g3;
  g3 = (b1 != g1 && b1 != g2) ? min(g3, b1) : g3;
  g3 = (b2 != g1 && b2 != g2) ? min(g3, b2) : g3;
  a1 = g1;
  a2 = g2;
  la = g3;
}

// Start of a job: the current centroids are the initial ones, the counters
// and statistics are zero, and center[j] is the mean of the initial centroids'
// coordinate j (0 where that is not finite), the shift the tensor-core pass
// applies to points and centroids alike (center null: not wanted).  One CTA per 32 dimensions.
constexpr int SETUP_THREADS = 1024;
__global__ void __launch_bounds__(SETUP_THREADS) km_setup_kernel(const float* __restrict__ init, uint32_t k,
                                                                 uint32_t d, float* __restrict__ c,
                                                                 float* __restrict__ center, unsigned long long* cnew,
                                                                 uint32_t* nflag, unsigned long long* stats) {
  __shared__ double red[SETUP_THREADS / 32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t j = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (j < d)
    for (uint32_t i = w; i < k; i += SETUP_THREADS / 32) {
      const float v = init[(uint64_t)i * d + j];
      c[(uint64_t)i * d + j] = v;
      s += (double)v;
    }
  red[w][lane] = s;
  __syncthreads();
  if (w == 0 && j < d) {
    for (int i = 1; i < SETUP_THREADS / 32; ++i) s += red[i][lane];
    const float m = (float)(s / (double)k);
    if (center) center[j] = isfinite(m) ? m : 0.f;
  }
  if (blockIdx.x == 0)
    for (uint32_t i = threadIdx.x; i < k; i += SETUP_THREADS) cnew[i] = 0;
  // counters, and the words behind the exponent (largest drift, sum of them)
  if (blockIdx.x == 0 && threadIdx.x < 24) nflag[threadIdx.x] = 0;
  if (blockIdx.x == 0 && threadIdx.x < 4) stats[threadIdx.x] = 0;
}

// FP32 assignment.  A CTA processes tiles of 64 points; warp w owns points
// 8w..8w+7 of the tile, lane l owns centroids l + 32 j (j < 8) of each chunk
// of up to 256 centroids.  Dot products accumulate over dimension chunks
// staged in shared memory (points transposed [dim][point], centroids
// [dim][centroid]).  When K <= 256 and D <= 64 the centroids are loaded once
// per CTA.
// KEYS (K <= 256): selection by packed keys (top-2 plus a lower bound of
// the other keys); else a float top-3 with indices.
template <bool KEYS>
__global__ void __launch_bounds__(KM_THREADS, 2)
km_assign_fp32_kernel(const float* __restrict__ x, uint32_t n, uint32_t d, const float* __restrict__ c, uint32_t k,
                      const float* __restrict__ cn, const unsigned int* cmax_bits, uint32_t* __restrict__ assign,
                      uint32_t* nchg, uint32_t* flagged, uint32_t* nflag, KmFew* __restrict__ pairs, uint32_t* npairs) {
  extern __shared__ float km_sm[];
  const int dc = d < DC_MAX ? (int)d : DC_MAX;
  const int kc = k < KC_MAX ? (int)k : KC_MAX;
  float* cs = km_sm;              // [dc][CS_LD]
  float* xs = km_sm + DC_MAX * CS_LD;  // [dc][XS_LD]
  __shared__ float nx_s[TP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t npts = n;
  const bool resident = k <= KC_MAX && d <= DC_MAX;
  const bool vec4 = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const float cmax = __uint_as_float(*cmax_bits);
  const float eps = 1.01f * (float)(d + 8) * 5.9604645e-8f;  // 2^-24

  auto load_c = [&](uint32_t k0, uint32_t d0) {
    for (int t = threadIdx.x; t < kc * dc; t += KM_THREADS) {
      const int kk = t / dc, dd = t % dc;
      const uint32_t kg = k0 + kk, dg = d0 + dd;
      cs[dd * CS_LD + kk] = (kg < k && dg < d) ? c[(uint64_t)kg * d + dg] : 0.f;
    }
  };
  if (resident) {
    load_c(0, 0);
    __syncthreads();
  }
  const uint32_t ntiles = (npts + TP - 1) / TP;
  uint32_t moved = 0;  // this lane's points that changed cluster
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint32_t p0 = tile * TP;
    Top3 tp[KEYS ? 1 : 8];
    uint32_t t1[KEYS ? 8 : 1], t2[KEYS ? 8 : 1];
    if (KEYS) {
#pragma unroll
      for (int i = 0; i < 8; ++i) t1[i] = t2[i] = KEY_NONE;
    } else {
#pragma unroll
      for (int i = 0; i < (KEYS ? 1 : 8); ++i) top3_init(tp[i]);
    }
    float nxacc = 0.f;  // ||x||^2 of point threadIdx.x (threads < TP), FMA over dims in order
    for (uint32_t k0 = 0; k0 < k; k0 += KC_MAX) {
      float acc[8][8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
      for (uint32_t d0 = 0; d0 < d; d0 += DC_MAX) {
        __syncthreads();
        if (!resident) load_c(k0, d0);
        const int dlim = (int)((d - d0) < (uint32_t)dc ? (d - d0) : (uint32_t)dc);
        // A warp item is 16 points x 8 dims: lane l loads point 16 (wi % 4) +
        // l % 16, dims 8 (wi / 4) + 4 (l / 16) .. + 3 (one 16-byte load when
        // rows allow), and stores them transposed; with the row stride TP + 4
        // the 32 lanes of each store hit 32 banks.
        for (int wi = warp; wi < (TP / 16) * ((dc + 7) / 8); wi += KM_THREADS / 32) {
          const int pp = 16 * (wi % (TP / 16)) + (lane & 15);
          const int dd = 8 * (wi / (TP / 16)) + 4 * (lane >> 4);
          const uint32_t pi = p0 + pp;
          float v[4] = {0.f, 0.f, 0.f, 0.f};
          if (pi < npts) {
            const uint32_t p = pi;
            const float* row = x + (uint64_t)p * d + d0 + dd;
            if (vec4 && dd + 4 <= dlim) {
              const float4 q = __ldg(reinterpret_cast<const float4*>(row));
              v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
            } else {
#pragma unroll
              for (int m = 0; m < 4; ++m)
                if (dd + m < dlim) v[m] = __ldg(row + m);
            }
          }
#pragma unroll
          for (int m = 0; m < 4; ++m)
            if (dd + m < dc) xs[(dd + m) * XS_LD + pp] = v[m];
        }
        __syncthreads();
        if (k0 == 0 && threadIdx.x < TP)
          for (int dd = 0; dd < dlim; ++dd)
            nxacc = fmaf(xs[dd * XS_LD + threadIdx.x], xs[dd * XS_LD + threadIdx.x], nxacc);
        for (int dd = 0; dd < dlim; ++dd) {
          const float4 xa = *reinterpret_cast<const float4*>(&xs[dd * XS_LD + warp * 8]);
          const float4 xb = *reinterpret_cast<const float4*>(&xs[dd * XS_LD + warp * 8 + 4]);
          const float xv[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
          float cv[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) cv[j] = cs[dd * CS_LD + lane + 32 * j];
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xv[i], cv[j], acc[i][j]);
        }
      }
      if (k0 == 0) {
        __syncthreads();
        if (threadIdx.x < TP) nx_s[threadIdx.x] = nxacc;
        __syncthreads();
      }
      // distances for this chunk
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t kk = k0 + lane + 32 * j;
        if (KEYS) {
          const bool valid = kk < k && lane + 32 * j < kc;
          const float ncv = valid ? cn[kk] : 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float dist = fmaf(-2.f, acc[i][j], nx_s[warp * 8 + i]) + ncv;
            top2_insert(t1[i], t2[i], valid ? dist_key(dist, kk) : KEY_NONE);
          }
        } else if (kk < k && lane + 32 * j < kc) {
          const float ncv = cn[kk];
#pragma unroll
          for (int i = 0; i < (KEYS ? 1 : 8); ++i) {
            const float dist = fmaf(-2.f, acc[i][j], nx_s[warp * 8 + i]) + ncv;
            top3_push(tp[i], dist, (int)kk);
          }
        }
      }
    }
    // combine the lanes' candidates for each of the warp's 8 points; lane i
    // then decides point i of the warp
    Top3 mt;
    top3_init(mt);
    if (KEYS) {
      uint32_t m1 = KEY_NONE, m2 = KEY_NONE, m3 = KEY_NONE;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        // a lane's keys other than its top-2 are all >= its second key
        uint32_t a1 = t1[i], a2 = t2[i], la = t2[i];
        for (int o = 16; o; o >>= 1) {
          const uint32_t b1 = __shfl_xor_sync(0xffffffffu, a1, o);
          const uint32_t b2 = __shfl_xor_sync(0xffffffffu, a2, o);
          const uint32_t lb = __shfl_xor_sync(0xffffffffu, la, o);
          top2lb_merge(a1, a2, la, b1, b2, lb);
        }
        if (lane == i) m1 = a1, m2 = a2, m3 = la;
      }
      // keys under-state a distance by less than 2^-15 of it: the margin
      // tests below get 2^-14 d1 more
      mt.d1 = key_dist(m1);
      mt.d2 = key_dist(m2);
      mt.d3 = key_dist(m3);
      mt.k1 = (int)(m1 & 0xFFu);
      mt.k2 = (int)(m2 & 0xFFu);
    } else {
#pragma unroll
      for (int i = 0; i < (KEYS ? 1 : 8); ++i) {
        for (int o = 16; o; o >>= 1) {
          Top3 ot;
          ot.d1 = __shfl_xor_sync(0xffffffffu, tp[i].d1, o);
          ot.d2 = __shfl_xor_sync(0xffffffffu, tp[i].d2, o);
          ot.d3 = __shfl_xor_sync(0xffffffffu, tp[i].d3, o);
          ot.k1 = __shfl_xor_sync(0xffffffffu, tp[i].k1, o);
          ot.k2 = __shfl_xor_sync(0xffffffffu, tp[i].k2, o);
          top3_merge(tp[i], ot);
        }
      }
#pragma unroll
      for (int i = 0; i < (KEYS ? 1 : 8); ++i)
        if (lane == i) mt = tp[i];
    }
    const uint32_t pi = p0 + warp * 8 + lane;
    bool flag = false, pair = false;
    if (lane < 8 && pi < npts) {
      const uint32_t p = pi;
      const float nxv = sqrtf(nx_s[warp * 8 + lane]);
      const float e = eps * (nxv + cmax) * (nxv + cmax);
      const float gap = 2.f * e + (KEYS ? 6.103515625e-05f * fmaxf(mt.d1, 0.f) : 0.f);
      // only the top two can be the exact minimum when the third is 2E away
      if (mt.d2 - mt.d1 > gap) {
        const uint32_t now = (uint32_t)mt.k1, old = nchg ? assign[p] & 0xffffu : now;
        assign[p] = km_word(now, old);
        moved += now != old;
      } else if (mt.d3 - mt.d1 > gap) pair = true;
      else flag = true;
    }
    const unsigned pm = __ballot_sync(0xffffffffu, pair);
    if (pm) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(npairs, (uint32_t)__popc(pm));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (pair) {
        const uint32_t p = pi;
        pairs[base + __popc(pm & ((1u << lane) - 1))] = km_few(p, (uint32_t)mt.k1 | ((uint32_t)mt.k2 << 12), 2);
      }
    }
    const unsigned fm = __ballot_sync(0xffffffffu, flag);
    if (fm) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(nflag, (uint32_t)__popc(fm));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (flag) {
        const uint32_t p = pi;
        flagged[base + __popc(fm & ((1u << lane) - 1))] = p;
      }
    }
  }
  moved = __reduce_add_sync(0xffffffffu, moved);
  if (lane == 0 && moved) atomicAdd(nchg, moved);
}

// Fixed-point exponent s (at most 60): the largest with max|x| 2^s < 2^39 and
// max|x| 2^s n < 2^62, so every q = rint(x 2^s) fits 40 bits (the update's
// hi/lo split) and no sum of n of them can overflow int64.  s may be
// negative for very large inputs; x 2^s then rounds only where it is far
// below 1/2, and rounds to 0 either way.  (max|x| = f 2^e with f < 1, so
// s <= 39 - e holds; n lowers it by at most 8 more.)
__device__ __forceinline__ int fx_shift_of(float m, uint32_t n) {
  if (!(m > 0.f)) return 60;
  const double lim = fmin(ldexp(1.0, 39), ldexp(1.0, 62) / (double)n);
  int e;
  frexpf(m, &e);
  int s = 39 - e < 60 ? 39 - e : 60;
  while (s > -200 && ldexp((double)m, s) >= lim) --s;
  return s;
}

// ------------------------------------------------- settling the near ties
// One kernel settles what the distance pass left open.
//
// Points with a few candidates (eight lanes each): FP32 direct differences to
// those centroids.  Their relative error is at most g =
// gamma_{D+3} for any summation order (Higham, eq. 3.5 on a sum of squares),
// so a ratio beyond widen decides the exact order.
//
// Listed points, in batches of SET_RP per CTA: FP32 direct differences to every
// centroid, one thread per centroid and all the batch's points at once: the
// points lie in shared memory dimension by dimension (one broadcast 16-byte
// read gives four points' coordinates), the centroids come from a transposed
// copy in coalesced reads that serve the whole batch, and two points go into
// each packed FP32 instruction.  Only the two smallest distances matter: when
// the second is beyond widen times the first, the first is the FP64 winner.
//
// A point that FP32 cannot decide is settled by the definition in FP64 on the
// spot: one with a few candidates by its eight lanes, a candidate each; a
// listed one by its whole CTA: the candidates are the centroids whose FP32
// distance is within the bound of the smallest; the products (x_j - c_j)^2,
// separately rounded, for all dimensions of a chunk of candidates at once
// (the FP64 pipe is narrow on this GPU), and one thread per candidate adding
// them with the dimensions in order.  (A point that equals a centroid needs no
// such choice: the difference of two unequal floats is not zero.)  The lowest index wins an exact tie;
// all-NaN distances give index 0, as the definition.
//
// Bounded by the FP32 pipe for long lists (2 K D operations a listed point)
// and by latency for short ones.  As three launches (pairs, a re-check with the
// centroids staged in each CTA's shared memory and one warp per point, a
// kernel for the FP64 points) this took 15 + 56 + 20 us at 4M x 64, K = 256
// (181K pairs, 22K listed points, 100 FP64 points); now 36 us.  For K x D
// beyond shared memory the re-check went warp by warp over the centroids: 531
// of 576 us at 250,000 x 128, K = 512; now 55 us (85 before the loads of a
// point's rows, word and bound, and of eight dimensions' centroids, went out
// together, and the CTAs with listed points left the others alone).
// stat[0] counts the points re-checked, stat[1] those settled in FP64.
constexpr int SET_RP = 16;        // listed points per batch
constexpr int SET_LD = SET_RP + 4;  // row stride of the staged points (16-byte rows)
constexpr int SET_T_MAX = 256;
constexpr uint32_t SET_PROD = 2048;  // doubles of product scratch
inline int set_threads(uint32_t k) { return k >= 225 ? 256 : (int)((k + 31) / 32 < 2 ? 64 : (k + 31) / 32 * 32); }
inline size_t set_smem(uint32_t d, uint32_t k) {
  const size_t stage = (size_t)d * SET_LD * 4, prod = (size_t)SET_PROD * 8;
  return (stage > prod ? stage : prod) + (size_t)d * 4 + (size_t)k * 8;
}
__device__ __forceinline__ float rel_bound_widen(uint32_t d) {
  const float g = 1.01f * (float)(d + 8) * 5.9604644775390625e-08f;
  return (1.f + g) / (1.f - g) * (1.f + 4.f * 5.9604644775390625e-08f);
}
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  return (unsigned long long)__float_as_uint(a) | ((unsigned long long)__float_as_uint(b) << 32);
}
// a += (x - c)^2 for two points at once (nc = {-c, -c}); x + (-c) rounds as x - c
__device__ __forceinline__ void sqdiff2(unsigned long long& a, unsigned long long x, unsigned long long nc) {
  unsigned long long t;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(x), "l"(nc));
  asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(a) : "l"(t));
}

struct SettleShared {
  uint32_t m1[SET_T_MAX / 32][SET_RP], k1[SET_T_MAX / 32][SET_RP], m2[SET_T_MAX / 32][SET_RP];
  uint32_t open[SET_RP];  // points of the batch left to FP64
  uint32_t nopen, ncand, moved;
  float red_f[SET_T_MAX / 32];
  double red_d[SET_T_MAX / 32];
  int red_k[SET_T_MAX / 32];
};

// The settled cluster of point p; has: its word holds the cluster of the round
// before (not in a job's first round).
__device__ __forceinline__ void settle_put(uint32_t* assign, uint32_t p, uint32_t now, bool has, uint32_t word,
                                           SettleShared& S) {
  const uint32_t old = has ? word & 0xffffu : now;
  assign[p] = km_word(now, old);
  if (now != old) atomicAdd(&S.moved, 1u);
}

// The FP64 definition for point p, by the whole CTA (all threads call this).
__device__ void settle_fp64(const float* __restrict__ x, uint32_t d, const float* __restrict__ c,
                            const float* __restrict__ ct, uint32_t k, uint32_t p, uint32_t* assign, bool has,
                            double* prod, float* xs, float* dist, uint32_t* cand, SettleShared& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const float widen = rel_bound_widen(d);
  const uint32_t cc = max(1u, min(SET_PROD / d, blockDim.x));  // candidates per product chunk (d <= 1024)
  const float* xp = x + (uint64_t)p * d;
  __syncthreads();  // the shared arrays' previous use is over
  for (uint32_t j = threadIdx.x; j < d; j += blockDim.x) xs[j] = xp[j];
  if (threadIdx.x == 0) S.ncand = 0;
  __syncthreads();
  float m = INFINITY;
  uint32_t same = 0x7fffffffu;  // the lowest centroid that is the point itself
  for (uint32_t kk = threadIdx.x; kk < k; kk += blockDim.x) {
    float s32 = 0.f;
    uint32_t bits = 0;
#pragma unroll 16
    for (uint32_t j = 0; j < d; ++j) {
      const float t = xs[j] - __ldg(ct + (uint64_t)j * k + kk);
      s32 = fmaf(t, t, s32);
      bits |= __float_as_uint(t);
    }
    dist[kk] = s32;
    m = fminf(m, s32);
    if (bits == 0) same = min(same, kk);
  }
  for (int o = 16; o; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
  same = __reduce_min_sync(0xffffffffu, same);
  if (lane == 0) S.red_f[warp] = m, S.red_k[warp] = (int)same;
  __syncthreads();
  float m32 = S.red_f[0];
  for (int w = 1; w < nw; ++w) m32 = fminf(m32, S.red_f[w]);
  for (int w = 0; w < nw; ++w) same = min(same, (uint32_t)S.red_k[w]);
  if (same != 0x7fffffffu) {  // its distance is zero, and no other's is less
    if (threadIdx.x == 0) settle_put(assign, p, same, has, has ? assign[p] : 0u, S);
    return;
  }
  const float lim = m32 * widen;
  for (uint32_t kk = threadIdx.x; kk < k; kk += blockDim.x)
    if (dist[kk] <= lim || m32 != m32) cand[atomicAdd(&S.ncand, 1u)] = kk;
  __syncthreads();
  const uint32_t nc = S.ncand;
  double best = INFINITY;
  int bk = 0x7fffffff;
  for (uint32_t c0 = 0; c0 < nc; c0 += cc) {
    const uint32_t cn = nc - c0 < cc ? nc - c0 : cc;
    for (uint32_t ci = warp; ci < cn; ci += nw) {
      const float* cp = c + (uint64_t)cand[c0 + ci] * d;
      for (uint32_t j = lane; j < d; j += 32) {
        const double t = __dsub_rn((double)xs[j], (double)__ldg(cp + j));
        prod[ci * d + j] = __dmul_rn(t, t);
      }
    }
    __syncthreads();
    if (threadIdx.x < cn) {
      double s64 = 0.0;
#pragma unroll 8
      for (uint32_t j = 0; j < d; ++j) s64 = __dadd_rn(s64, prod[threadIdx.x * d + j]);
      const int kk = (int)cand[c0 + threadIdx.x];
      if (s64 < best || (s64 == best && kk < bk)) best = s64, bk = kk;
    }
    __syncthreads();
  }
  for (int o = 16; o; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
    if (ob < best || (ob == best && ok < bk)) best = ob, bk = ok;
  }
  if (lane == 0) S.red_d[warp] = best, S.red_k[warp] = bk;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < nw; ++w)
      if (S.red_d[w] < best || (S.red_d[w] == best && S.red_k[w] < bk)) best = S.red_d[w], bk = S.red_k[w];
    settle_put(assign, p, bk == 0x7fffffff ? 0u : (uint32_t)bk, has, has ? assign[p] : 0u, S);
  }
}

__device__ __forceinline__ uint32_t few_cand(const KmFew& e, uint32_t i) {
  return (uint32_t)(((uint64_t)e.lo | ((uint64_t)e.hi << 32)) >> (12 * i)) & 0xFFFu;
}
// FP32 squared distances of an entry's first M candidates, by eight lanes
// (lane sl of them): every candidate's row and the point's are read together,
// 16 bytes a lane where rows allow (vec).  All 32 lanes call this.
template <int M>
__device__ __forceinline__ void few_dists(const float* __restrict__ x, const float* __restrict__ c, uint32_t d,
                                          const KmFew& e, uint32_t nc, uint32_t sl, bool vec,
                                          float (&f)[KM_CAND_MAX]) {
  const float* xp = x + (uint64_t)e.p * d;
  const float* cp[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    cp[i] = c + (uint64_t)few_cand(e, (uint32_t)i < nc ? i : 0) * d;
    f[i] = 0.f;
  }
  if (nc == 0) {
  } else if (vec) {
    for (uint32_t j = 4 * sl; j < d; j += 32) {
      const float4 xv = __ldg(reinterpret_cast<const float4*>(xp + j));
#pragma unroll
      for (int i = 0; i < M; ++i) {
        const float4 cv = __ldg(reinterpret_cast<const float4*>(cp[i] + j));
        const float t0 = xv.x - cv.x, t1 = xv.y - cv.y, t2 = xv.z - cv.z, t3 = xv.w - cv.w;
        f[i] = fmaf(t0, t0, fmaf(t1, t1, fmaf(t2, t2, fmaf(t3, t3, f[i]))));
      }
    }
  } else {
    for (uint32_t j = sl; j < d; j += 8) {
      const float xv = __ldg(xp + j);
#pragma unroll
      for (int i = 0; i < M; ++i) {
        const float t = xv - __ldg(cp[i] + j);
        f[i] = fmaf(t, t, f[i]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int o = 4; o; o >>= 1) f[i] += __shfl_xor_sync(0xffffffffu, f[i], o);
}

__device__ __forceinline__ KmFew load_few(const KmFew* __restrict__ few, uint32_t n, uint64_t i) {
  return i < n ? few[i] : KmFew{0, 0, 0};
}

// MULTI: more centroids than threads, so each thread keeps a running top-2.
// With maxabs not null (the first iteration, whose distance pass or a pass
// before it found max |x|) one thread also sets the update's exponent.
template <bool MULTI>
__global__ void __launch_bounds__(SET_T_MAX) km_settle_kernel(
    const float* __restrict__ x, uint32_t n, uint32_t d, const float* __restrict__ c, const float* __restrict__ ct,
    uint32_t k, const KmFew* __restrict__ pairs, const uint32_t* npairs, const uint32_t* __restrict__ list,
    const uint32_t* nlist, uint32_t* assign, uint32_t* nchg, unsigned long long* stat, const unsigned int* maxabs, int* shift,
    unsigned int* cmax_next, KmBounds B) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char set_sm[];
  __shared__ SettleShared S;
  const size_t stage = (size_t)d * SET_LD * 4;
  float* xt = reinterpret_cast<float*>(set_sm);       // [d][SET_LD] staged points, or
  double* prod = reinterpret_cast<double*>(set_sm);   // [cc][d] FP64 products
  float* xs = reinterpret_cast<float*>(set_sm + (stage > SET_PROD * 8 ? stage : SET_PROD * 8));  // [d]
  float* dist = xs + d;                               // [k]
  uint32_t* cand = reinterpret_cast<uint32_t*>(dist + k);  // [k]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t np = *npairs, nf = *nlist;
  if (threadIdx.x == 0) S.moved = 0;
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (maxabs) *shift = fx_shift_of(__uint_as_float(*maxabs), n);
    *cmax_next = 0;  // the next iteration's max ||c||
    if (np + nf) atomicAdd(stat, (unsigned long long)np + nf);
  }
  const float widen = rel_bound_widen(d);
  const bool bounds = km_keeps_bounds(B);
  const bool vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const uint64_t rb = ((uint64_t)nf + SET_RP - 1) / SET_RP;
  unsigned long long settled = 0;  // points settled in FP64
  // the few-candidate points: warps on their own, four points at a time.  The
  // CTAs that have a batch of listed points leave them to the others (up to
  // half of the CTAs), so that no CTA's chain of loads holds both.
  const uint32_t lead = (uint32_t)(rb < gridDim.x / 2 ? rb : gridDim.x / 2);
  if (blockIdx.x >= lead) {
    const uint32_t sl = lane & 7;
    const uint64_t w0 = (uint64_t)(blockIdx.x - lead) * nw + warp, ws = (uint64_t)(gridDim.x - lead) * nw;
    KmFew next = load_few(pairs, np, 4 * w0 + (lane >> 3));
    for (uint64_t f0 = 4 * w0; f0 < np; f0 += 4 * ws) {
      const KmFew e = next;
      next = load_few(pairs, np, f0 + 4 * ws + (lane >> 3));
      // (loaded with the rows, not after them)
      const uint32_t word = nchg ? assign[e.p] : 0u;
      const float l = bounds ? B.lb[e.p] : 0.f;
      const uint32_t nc = e.hi >> 28;
      float fd[KM_CAND_MAX];
      if (__any_sync(0xffffffffu, nc > 2)) few_dists<KM_CAND_MAX>(x, c, d, e, nc, sl, vec, fd);
      else few_dists<2>(x, c, d, e, nc, sl, vec, fd);
      float m1 = INFINITY, m2 = INFINITY;
      uint32_t k1 = 0;
#pragma unroll
      for (uint32_t i = 0; i < KM_CAND_MAX; ++i)
        if (i < nc) {
          if (fd[i] < m1) m2 = m1, m1 = fd[i], k1 = few_cand(e, i);
          else if (!(fd[i] >= m2)) m2 = fd[i];  // (a NaN makes m2 NaN: the point is left to FP64)
        }
      const bool clear = nc == 0 || m2 > m1 * widen;
      if (!__all_sync(0xffffffffu, clear)) {
        // the definition, one candidate per lane, dimensions in order
        double best = INFINITY;
        uint32_t bk = 0xffffffffu;
        if (!clear && sl < nc) {
          bk = few_cand(e, sl);
          const float* xp = x + (uint64_t)e.p * d;
          const float* cp = c + (uint64_t)bk * d;
          double s64 = 0.0;
#pragma unroll 8
          for (uint32_t j = 0; j < d; ++j) {
            const double t = __dsub_rn((double)__ldg(xp + j), (double)__ldg(cp + j));
            s64 = __dadd_rn(s64, __dmul_rn(t, t));
          }
          best = s64;
          if (best != best) best = INFINITY, bk = 0xffffffffu;  // NaN never wins
        }
#pragma unroll
        for (int o = 4; o; o >>= 1) {
          const double ob = __shfl_xor_sync(0xffffffffu, best, o);
          const uint32_t ok = __shfl_xor_sync(0xffffffffu, bk, o);
          if (ob < best || (ob == best && ok < bk)) best = ob, bk = ok;
        }
        if (!clear && sl == 0) {
          settle_put(assign, e.p, bk == 0xffffffffu ? 0u : bk, nchg, word, S);
          if (bounds) B.ub[e.p] = INFINITY;  // no bounds: the next round computes it again
          ++settled;
        }
      }
      if (clear && nc && sl == 0) {
        settle_put(assign, e.p, k1, nchg, word, S);
        if (bounds) {  // the distance pass left the bound of the other centroids
          km_put_bounds(B, e.p, B.drift[k1], *B.far, m1 * widen + 1e-36f,
                        fminf(m2 * (2.f - widen) - 1e-36f, l * l * 0.999999f));
        }
      }
    }
  }
  for (uint64_t b = blockIdx.x; b < rb; b += gridDim.x) {
    __syncthreads();  // the previous batch's shared arrays are no longer read
    if (threadIdx.x == 0) S.nopen = 0;
    {
      const uint32_t f0 = (uint32_t)b * SET_RP;
      const uint32_t cnt = nf - f0 < (uint32_t)SET_RP ? nf - f0 : (uint32_t)SET_RP;
      for (uint32_t r = warp; r < (uint32_t)SET_RP; r += nw) {
        const float* xp = x + (uint64_t)list[f0 + (r < cnt ? r : 0)] * d;
        for (uint32_t j = lane; j < d; j += 32) xt[j * SET_LD + r] = xp[j];
      }
      __syncthreads();
      uint32_t b1[MULTI ? SET_RP : 1], bi[MULTI ? SET_RP : 1], b2[MULTI ? SET_RP : 1];
      if (MULTI) {
#pragma unroll
        for (int r = 0; r < (MULTI ? SET_RP : 1); ++r) b1[r] = b2[r] = 0x7F800000u, bi[r] = 0;
      }
      unsigned long long acc[SET_RP / 2];
      for (uint32_t kk = threadIdx.x; MULTI ? kk - threadIdx.x < k : kk == threadIdx.x; kk += blockDim.x) {
#pragma unroll
        for (int q = 0; q < SET_RP / 2; ++q) acc[q] = 0ull;
        if (kk < k) {
#pragma unroll 8
          for (uint32_t j = 0; j < d; ++j) {
            const float cv = -__ldg(ct + (uint64_t)j * k + kk);
            const unsigned long long nc = pack2(cv, cv);
            const ulonglong2* row = reinterpret_cast<const ulonglong2*>(xt + j * SET_LD);
#pragma unroll
            for (int q = 0; q < SET_RP / 4; ++q) {
              const ulonglong2 v = row[q];
              sqdiff2(acc[2 * q], v.x, nc);
              sqdiff2(acc[2 * q + 1], v.y, nc);
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < SET_RP / 2; ++q) acc[q] = 0x7F8000007F800000ull;  // no centroid: +inf
        }
        if (MULTI) {
#pragma unroll
          for (int r = 0; r < (MULTI ? SET_RP : 1); ++r) {
            const uint32_t v = (uint32_t)(acc[r >> 1] >> (32 * (r & 1)));
            if (v < b1[r]) b2[r] = b1[r], b1[r] = v, bi[r] = kk;
            else b2[r] = min(b2[r], v);
          }
        }
      }
      // distances are non-negative (or NaN, above every other), so their bits order like them
#pragma unroll
      for (int r = 0; r < SET_RP; ++r) {
        const uint32_t v = MULTI ? b1[MULTI ? r : 0] : (uint32_t)(acc[r >> 1] >> (32 * (r & 1)));
        const uint32_t m1 = __reduce_min_sync(0xffffffffu, v);
        const int lead = __ffs(__ballot_sync(0xffffffffu, v == m1)) - 1;
        const uint32_t m2 =
            __reduce_min_sync(0xffffffffu, lane == lead ? (MULTI ? b2[MULTI ? r : 0] : 0x7F800000u) : v);
        if (lane == lead) {
          S.m1[warp][r] = m1;
          S.m2[warp][r] = m2;
          S.k1[warp][r] = MULTI ? bi[MULTI ? r : 0] : threadIdx.x;
        }
      }
      __syncthreads();
      if (threadIdx.x < cnt) {
        const uint32_t r = threadIdx.x;
        uint32_t m1 = S.m1[0][r], k1 = S.k1[0][r], m2 = S.m2[0][r];
        for (int w = 1; w < nw; ++w) {
          const uint32_t o1 = S.m1[w][r];
          if (o1 < m1) m2 = min(m1, S.m2[w][r]), m1 = o1, k1 = S.k1[w][r];
          else m2 = min(m2, o1);
        }
        const uint32_t p = list[f0 + r];
        if (__uint_as_float(m2) > __uint_as_float(m1) * widen) {
          settle_put(assign, p, k1, nchg, nchg ? assign[p] : 0u, S);
          if (bounds)
            km_put_bounds(B, p, B.drift[k1], *B.far, __uint_as_float(m1) * widen + 1e-36f,
                          __uint_as_float(m2) * (2.f - widen) - 1e-36f);
        } else {
          S.open[atomicAdd(&S.nopen, 1u)] = p;
        }
      }
    }
    __syncthreads();
    const uint32_t no = S.nopen;
    if (bounds && threadIdx.x < no) B.ub[S.open[threadIdx.x]] = INFINITY;  // no bounds: the next round computes it again
    for (uint32_t i = 0; i < no; ++i) settle_fp64(x, d, c, ct, k, S.open[i], assign, nchg, prod, xs, dist, cand, S);
    if (threadIdx.x == 0) settled += no;
  }
  if (settled) atomicAdd(stat + 1, settled);
  __syncthreads();
  if (threadIdx.x == 0 && S.moved) atomicAdd(nchg, S.moved);
}

// max |x| over all coordinates (as float bits; non-negative floats order like ints)
__global__ void km_maxabs_kernel(const float* __restrict__ x, uint64_t cnt, unsigned int* out) {
  unsigned int m = 0;
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
  uint64_t done = 0;
  if (((uintptr_t)x & 15) == 0) {
    const uint64_t n4 = cnt / 4;
    const float4* x4 = reinterpret_cast<const float4*>(x);
    for (uint64_t i = tid; i < n4; i += nth) {
      const float4 v = __ldg(x4 + i);
      m = max(m, max(max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))),
                     max(__float_as_uint(fabsf(v.z)), __float_as_uint(fabsf(v.w)))));
    }
    done = n4 * 4;
  }
  for (uint64_t i = done + tid; i < cnt; i += nth) m = max(m, __float_as_uint(fabsf(x[i])));
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__device__ __forceinline__ uint32_t cluster_of(const uint32_t* assign, uint64_t i, uint32_t k) {
  return km_now(assign[i], k);
}

// ------------------------------------------------------- update by changes
// After the first rounds few points change cluster (0.2 - 5% a round on
// Gaussian mixtures from the third round on), and the sums are exact integers:
// subtracting a moved point from its old cluster and adding it to its new one
// gives the same sums, bit for bit, as adding all points again.  When few
// points moved (at most lim), the update kernels do only that: they read the
// assignment words (4 bytes a point instead of 4 D + 4) and issue two 64-bit
// global adds per coordinate of each moved point; otherwise they add all
// points, as in the first round.  Which one is decided on the device, by every
// kernel of the update alike, from the count the distance and settle passes
// left (chg null: the first round).
//
// The line: n / 4 beside the window-sorted update, whose CTAs collect the
// changes in their shared-memory sums, unless at most n / 256 points moved
// (4M x 64, K = 256: all points 186 us; 21% moved 183 us (the ten rounds 30 us
// shorter than with n / 8), 1.8% 49 us and 124
// straight to the global sums, 0.6% 32 us; 0.2% 17 us straight); n / 32 beside
// the other local-array updates; n / 8 beside the sorted update (250,000 x 128,
// K = 512: all points 107 us, 4.1% moved 27 us, 2.3% 20 us).
constexpr uint32_t KM_DELTA_WINDOW = 4, KM_DELTA_DIRECT = 256, KM_DELTA_LOCAL = 32, KM_DELTA_SORTED = 8;
__device__ __forceinline__ bool km_by_changes(const uint32_t* chg, uint32_t lim) { return chg && *chg <= lim; }

__device__ __forceinline__ void lq_split(float v, int& hi, int& lo);

// The whole grid's moved points (every thread of every CTA calls this): a warp
// takes 128 consecutive words, 16 bytes a lane, and up to KM_DELTA_ROWS moved
// points' rows at a time.
constexpr int KM_DELTA_ROWS = 4;
__device__ __forceinline__ void km_apply_changes(const float* __restrict__ x, uint32_t n, uint32_t d, uint32_t k,
                                                 uint32_t* assign, const int* shift, long long* sums,
                                                 unsigned long long* counts) {
  const int lane = threadIdx.x & 31;
  const float scale = ldexpf(1.f, *shift);
  const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long* S = reinterpret_cast<unsigned long long*>(sums);
  for (uint64_t b = w0 * 128; b < n; b += nw * 128) {
    uint32_t wd[4];
    const uint64_t i0 = b + 4 * (uint64_t)lane;
    if (i0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(assign + i0);
      wd[0] = v.x, wd[1] = v.y, wd[2] = v.z, wd[3] = v.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) wd[q] = i0 + q < n ? assign[i0 + q] : 0u;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t to = km_now(wd[q], k), from = km_summed(wd[q], k);
      const bool moved = to != from;
      if (moved) {
        assign[i0 + q] = km_word(to, to);
        atomicAdd(counts + to, 1ull);
        atomicAdd(counts + from, ~0ull);
      }
      unsigned m = __ballot_sync(0xffffffffu, moved);
      while (m) {
        uint64_t row[KM_DELTA_ROWS];
        uint32_t t[KM_DELTA_ROWS], f[KM_DELTA_ROWS];
        bool on[KM_DELTA_ROWS];
#pragma unroll
        for (int u = 0; u < KM_DELTA_ROWS; ++u) {
          const int src = m ? __ffs(m) - 1 : 0;
          on[u] = m != 0;
          m &= m - 1;
          row[u] = (b + 4 * (uint64_t)src + q) * d;
          t[u] = __shfl_sync(0xffffffffu, to, src) * d;
          f[u] = __shfl_sync(0xffffffffu, from, src) * d;
        }
        for (uint32_t j = lane; j < d; j += 32) {
          float v[KM_DELTA_ROWS];
#pragma unroll
          for (int u = 0; u < KM_DELTA_ROWS; ++u) v[u] = on[u] ? __ldg(x + row[u] + j) : 0.f;
#pragma unroll
          for (int u = 0; u < KM_DELTA_ROWS; ++u) {
            if (!on[u]) break;
            int hi, lo;
            lq_split(v[u] * scale, hi, lo);
            const long long qv = (long long)hi * (1ll << 20) + (long long)lo;
            if (qv) {
              atomicAdd(S + t[u] + j, (unsigned long long)qv);
              atomicAdd(S + f[u] + j, (unsigned long long)-qv);
            }
          }
        }
      }
    }
  }
}
// Before a full update: the words' old clusters become the new ones.
__device__ __forceinline__ void km_settle_word(uint32_t* assign, uint64_t i, uint32_t k) {
  const uint32_t w = assign[i], c = km_now(w, k);
  if (w != km_word(c, c)) assign[i] = km_word(c, c);
}

// First kernel of the sorted update: cluster sizes (a CTA counts in shared
// memory, then adds to the global counts), and clears the sums; or the whole
// update by changes.
__global__ void km_count_kernel(const float* __restrict__ x, uint32_t d, uint32_t* __restrict__ assign, uint32_t n,
                                uint32_t k, unsigned long long* counts, unsigned long long* cnew, const uint32_t* chg, uint32_t lim,
                                const int* shift, long long* sums) {
  pdl_wait();
  if (km_by_changes(chg, lim)) {
    km_apply_changes(x, n, d, k, assign, shift, sums, counts);
    return;
  }
  extern __shared__ uint32_t hc[];
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, nth = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = tid; i < (uint64_t)k * d; i += nth) sums[i] = 0;
  for (uint32_t t = threadIdx.x; t < k; t += blockDim.x) hc[t] = 0;
  __syncthreads();
  for (uint64_t i = tid; i < n; i += nth) {
    km_settle_word(assign, i, k);
    atomicAdd(&hc[cluster_of(assign, i, k)], 1u);
  }
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < k; t += blockDim.x)
    if (hc[t]) atomicAdd(cnew + t, (unsigned long long)hc[t]);
}

// Exclusive scan of the counts into each cluster's write cursor (one CTA).
__global__ void km_offsets_kernel(const unsigned long long* counts, uint32_t k, uint32_t* cursor, const uint32_t* chg, uint32_t lim) {
  pdl_wait();
  if (km_by_changes(chg, lim)) return;
  __shared__ uint32_t carry;
  __shared__ uint32_t wsum[32];
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t b = 0; b < k; b += blockDim.x) {
    const uint32_t i = b + threadIdx.x;
    const uint32_t v = i < k ? (uint32_t)counts[i] : 0;
    uint32_t incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
      uint32_t wi = w;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += t;
      }
      wsum[lane] = wi - w;
    }
    __syncthreads();
    const uint32_t ex = carry + wsum[warp] + incl - v;
    if (i < k) cursor[i] = ex;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = ex + v;
    __syncthreads();
  }
}

// Counting-sort scatter: perm lists the points grouped by cluster (order
// inside a cluster does not matter: the sums are exact integers).  A CTA takes
// a chunk of points, counts them per cluster in shared memory, reserves each
// cluster's range with one global atomic, then places its points with
// shared-memory cursors.
constexpr int SCAT_THREADS = 256;
constexpr int SCAT_PER_THREAD = 16;
__global__ void __launch_bounds__(SCAT_THREADS) km_scatter_kernel(const uint32_t* __restrict__ assign, uint32_t n,
                                                                  uint32_t k, uint32_t* cursor,
                                                                  uint32_t* __restrict__ perm, const uint32_t* chg, uint32_t lim) {
  pdl_wait();
  if (km_by_changes(chg, lim)) return;
  extern __shared__ uint32_t sc[];  // [k] local counts, then local cursors
  const uint64_t chunk = (uint64_t)SCAT_THREADS * SCAT_PER_THREAD;
  const uint64_t b0 = (uint64_t)blockIdx.x * chunk;
  for (uint32_t t = threadIdx.x; t < k; t += SCAT_THREADS) sc[t] = 0;
  __syncthreads();
  uint32_t a[SCAT_PER_THREAD];
#pragma unroll
  for (int r = 0; r < SCAT_PER_THREAD; ++r) {
    const uint64_t i = b0 + (uint64_t)r * SCAT_THREADS + threadIdx.x;
    a[r] = i < n ? cluster_of(assign, i, k) : 0xffffffffu;
    if (a[r] != 0xffffffffu) atomicAdd(&sc[a[r]], 1u);
  }
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < k; t += SCAT_THREADS)
    if (sc[t]) sc[t] = atomicAdd(cursor + t, sc[t]);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < SCAT_PER_THREAD; ++r) {
    const uint64_t i = b0 + (uint64_t)r * SCAT_THREADS + threadIdx.x;
    if (a[r] != 0xffffffffu) perm[atomicAdd(&sc[a[r]], 1u)] = (uint32_t)i;
  }
}

// Per-cluster int64 fixed-point sums.  Warp w adds points perm[64w ..
// 64w+63]; they come in runs of one cluster (ends[c] = one past the last
// position of cluster c in perm, so a run's cluster needs no lookup of the
// point's assignment), summed in registers (lane l holds dimensions l and
// l+32 of the current 64-dimension slice) and added to the global sums once
// per run.  Eight rows are in flight per warp.
constexpr int SUM_RUN = 64;
constexpr int SUM_UNROLL = 8;
// Round-half-even of a finite FP32 value to int64 with FP32 adds and integer
// operations only: the FP32 -> int64 conversion instruction issues on the FP64
// pipe, which is narrow on this GPU and became the sum kernel's limit.
//   |v| < 2^22:  v + 1.5*2^23 rounds (ties to even) to an integer whose value
//                minus 1.5*2^23 sits in the low bits of the sum's encoding;
//   |v| >= 2^23: v is an integer, its significand shifted by e - 150;
//   in between:  one fraction bit, rounded to even by hand.
__device__ __forceinline__ long long rint_i64(float v) {
  const uint32_t b = __float_as_uint(v);
  const uint32_t e = (b >> 23) & 0xFFu;
  if (e < 149u) return (long long)(int32_t)(__float_as_uint(__fadd_rn(v, 12582912.f)) - 0x4B400000u);
  const uint64_t m = (b & 0x7FFFFFu) | 0x800000u;
  const uint64_t q = e == 149u ? (m >> 1) + (m & (m >> 1) & 1u) : m << ((e - 150u) & 63u);
  return (b >> 31) ? -(long long)q : (long long)q;
}
__device__ __forceinline__ void sum_flush(long long* sums, uint32_t cur, uint32_t d, uint32_t dj0, uint32_t dj1,
                                          long long a0, long long a1) {
  if (dj0 < d && a0) atomicAdd(reinterpret_cast<unsigned long long*>(sums + (uint64_t)cur * d + dj0), (unsigned long long)a0);
  if (dj1 < d && a1) atomicAdd(reinterpret_cast<unsigned long long*>(sums + (uint64_t)cur * d + dj1), (unsigned long long)a1);
}
__global__ void __launch_bounds__(256) km_sum_kernel(const float* __restrict__ x, uint32_t n, uint32_t d, uint32_t k,
                                                     const uint32_t* __restrict__ ends,
                                                     const uint32_t* __restrict__ perm, const int* shift,
                                                     long long* sums, const uint32_t* chg, uint32_t lim) {
  pdl_wait();
  if (km_by_changes(chg, lim)) return;
  const int lane = threadIdx.x & 31;
  const uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t p0 = w * SUM_RUN;
  if (p0 >= n) return;
  const uint64_t p1 = (p0 + SUM_RUN) < n ? p0 + SUM_RUN : n;
  // x * 2^s is exact in FP32 (a power-of-two scale far from overflow), so
  // rounding it to int64 gives the same q as in double precision
  const float scale = ldexpf(1.f, *shift);
  uint32_t idx[2];
  idx[0] = perm[p0 + lane < p1 ? p0 + lane : p0];
  idx[1] = perm[p0 + 32 + lane < p1 ? p0 + 32 + lane : p0];
  // cluster of position p0: the first c with ends[c] > p0
  uint32_t c0 = 0, hi = k - 1;
  while (c0 < hi) {
    const uint32_t mid = (c0 + hi) >> 1;
    if (ends[mid] > p0) hi = mid;
    else c0 = mid + 1;
  }
  for (uint32_t j0 = 0; j0 < d; j0 += 64) {
    const uint32_t dj0 = j0 + lane, dj1 = j0 + 32 + lane;
    long long a0 = 0, a1 = 0;
    uint32_t cur = c0, cend = ends[c0];
    for (uint64_t p = p0; p < p1; p += SUM_UNROLL) {
      float v[SUM_UNROLL][2];
#pragma unroll
      for (int u = 0; u < SUM_UNROLL; ++u) {
        const uint64_t pp = p + u;
        const uint32_t sel = (uint32_t)(pp - p0);
        const uint32_t i = __shfl_sync(0xffffffffu, sel < 32 ? idx[0] : idx[1], (int)(sel & 31));
        const bool ok = pp < p1;
        v[u][0] = (ok && dj0 < d) ? x[(uint64_t)i * d + dj0] : 0.f;
        v[u][1] = (ok && dj1 < d) ? x[(uint64_t)i * d + dj1] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < SUM_UNROLL; ++u) {
        const uint64_t pp = p + u;
        if (pp >= p1) break;
        while (pp >= cend) {  // warp-uniform: the run of cluster cur ended (empty clusters skipped)
          sum_flush(sums, cur, d, dj0, dj1, a0, a1);
          a0 = a1 = 0;
          ++cur;
          cend = ends[cur];
        }
        a0 += rint_i64(v[u][0] * scale);
        a1 += rint_i64(v[u][1] * scale);
      }
    }
    sum_flush(sums, cur, d, dj0, dj1, a0, a1);
  }
}

// Update step with local arrays (Sec. III-E: the array container, privatised
// per thread block).  A CTA's [k][d] fixed-point sums and [k] counts live in
// shared memory; one CTA per SM streams a contiguous range of points in input
// order (coalesced rows: no sort and no gather) and adds each coordinate with
// shared-memory atomics.  A 64-bit sum is kept as two 32-bit words, each
// added by a native 32-bit atomic: the low word's add returns the old value,
// and a carry out of it (new < old) goes into the high word's add, so
// hi * 2^32 + lo is the exact sum modulo 2^64 (which holds it: the scale
// keeps |sum| below 2^62).  The CTA then stores its sums as one partial
// (plain stores) and adds its counts to the global counts;
// km_finalize_kernel adds the partials.  Integer sums make the result
// independent of the order.
__device__ __forceinline__ void add64_split(uint32_t* lo, uint32_t* hi, long long q) {
  const uint32_t ql = (uint32_t)q;
  const uint32_t old = atomicAdd(lo, ql);
  atomicAdd(hi, (uint32_t)((unsigned long long)q >> 32) + (old + ql < old ? 1u : 0u));
}
constexpr int LS_THREADS = 1024;
constexpr int LS_ROWS = 4;  // rows in flight per warp
constexpr uint32_t LS_MAX_CTAS = 160;  // partials held in scratch
constexpr uint64_t LS_SMEM_MAX = 200 * 1024;
inline bool local_sums_fit(uint64_t d, uint64_t k) { return k * d * 8 + k * 4 <= LS_SMEM_MAX; }
__global__ void __launch_bounds__(LS_THREADS, 1) km_local_sum_kernel(const float* __restrict__ x, uint32_t n,
                                                                     uint32_t d, uint32_t k,
                                                                     uint32_t* __restrict__ assign,
                                                                     const int* shift, long long* __restrict__ part,
                                                                     unsigned long long* counts,
                                                                     unsigned long long* cnew, const uint32_t* chg, uint32_t lim,
                                                                     long long* sums) {
  pdl_wait();
  if (km_by_changes(chg, lim)) {
    km_apply_changes(x, n, d, k, assign, shift, sums, counts);
    return;
  }
  extern __shared__ __align__(16) unsigned char ls_sm[];
  const uint64_t kd = (uint64_t)k * d;
  uint32_t* SL = reinterpret_cast<uint32_t*>(ls_sm);  // low words [k][d]
  uint32_t* SH = SL + kd;                             // high words [k][d]
  unsigned int* C = SH + kd;
  for (uint64_t i = threadIdx.x; i < 2 * kd; i += LS_THREADS) SL[i] = 0;
  for (uint32_t i = threadIdx.x; i < k; i += LS_THREADS) C[i] = 0;
  __syncthreads();
  const float scale = ldexpf(1.f, *shift);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t per = (((uint64_t)n + gridDim.x - 1) / gridDim.x + 31) & ~31ull;
  const uint64_t p0 = (uint64_t)blockIdx.x * per;
  const uint64_t p1 = p0 + per < (uint64_t)n ? p0 + per : (uint64_t)n;
  for (uint64_t r0 = p0 + 32 * (uint64_t)warp; r0 < p1; r0 += 32 * (LS_THREADS / 32)) {
    // 32 consecutive rows per warp step; lane j holds row r0 + j's cluster
    const uint32_t nr = (uint32_t)(p1 - r0 < 32 ? p1 - r0 : 32);
    if ((uint32_t)lane < nr) km_settle_word(assign, r0 + lane, k);
    const uint32_t cl = (uint32_t)lane < nr ? cluster_of(assign, r0 + lane, k) : 0u;
    if ((uint32_t)lane < nr) atomicAdd(&C[cl], 1u);
    for (uint32_t j0 = 0; j0 < d; j0 += 64) {
      const uint32_t dj0 = j0 + lane, dj1 = j0 + 32 + lane;
      for (uint32_t rr = 0; rr < nr; rr += LS_ROWS) {
        float v[LS_ROWS][2];
        uint32_t c[LS_ROWS];
#pragma unroll
        for (int u = 0; u < LS_ROWS; ++u) {
          const uint32_t j = rr + u;
          c[u] = __shfl_sync(0xffffffffu, cl, (int)(j & 31));
          const bool ok = j < nr;
          const float* row = x + (r0 + j) * d;
          v[u][0] = (ok && dj0 < d) ? row[dj0] : 0.f;
          v[u][1] = (ok && dj1 < d) ? row[dj1] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < LS_ROWS; ++u) {
          if (rr + u >= nr) break;  // warp-uniform
          const uint32_t b = c[u] * d;
          if (dj0 < d) add64_split(SL + b + dj0, SH + b + dj0, rint_i64(v[u][0] * scale));
          if (dj1 < d) add64_split(SL + b + dj1, SH + b + dj1, rint_i64(v[u][1] * scale));
        }
      }
    }
  }
  __syncthreads();
  long long* P = part + (uint64_t)blockIdx.x * kd;
  for (uint64_t i = threadIdx.x; i < kd; i += LS_THREADS)
    P[i] = (long long)(((unsigned long long)SH[i] << 32) | SL[i]);
  for (uint32_t i = threadIdx.x; i < k; i += LS_THREADS)
    if (C[i]) atomicAdd(cnew + i, (unsigned long long)C[i]);
}

// Pipelined form of the local-array update, for rows of a multiple of 4
// floats starting 16-byte aligned.  Warp 0 is the producer: its lane 0
// streams chunks of `rows` consecutive points and their cluster ids into an
// LP_ST-deep shared-memory ring with bulk copies (completion counted on one
// mbarrier per stage) and refills a stage as soon as every worker warp has
// released it; warps 1..31 are workers, warp w taking rows w - 1, w - 1 +
// 31, ... of each chunk.  (With a worker refilling the ring only after its
// own rows, the ring ran dry and the kernel waited on DRAM latency.)
//
// Exact sums without 64-bit shared atomics.  The scale keeps |x 2^s| < 2^39
// (fx_shift_of), so q = rint(x 2^s) = hi 2^20 + lo with hi, lo integers
// of magnitude <= 2^19, both formed by FP32 adds that are exact (lq_split);
// each goes into a 32-bit shared-memory array with a non-returning add.
// Within a window of at most LP_FLUSH_ROWS points no 32-bit sum can overflow,
// so after each window the workers add hi 2^20 + lo of every (cluster, dim)
// into the CTA's own int64 partial in global memory (plain read-modify-
// write: no other CTA touches it) and clear the arrays.  Integer sums stay
// exact and order-independent, equal to the sum of rint(x 2^s) formed any
// other way.
//
// Every wait is bounded.  Workers run the same chunks and barriers whatever
// happens; after a wait gives up, chunks are skipped and the producer issues
// no more copies (it issues into a stage only after every worker released
// the stage's previous chunk with no error raised, i.e. after that chunk
// landed), lets the last copies it issued land, and the CTA counts itself in
// *timeouts.
constexpr int LP_ST = 4;
constexpr int LP_WORKERS = LS_THREADS / 32 - 1;  // warp 0 produces
constexpr uint32_t LP_CHUNK_MAX = 24 * 1024;     // bytes of points per stage, at most
constexpr uint32_t LP_FLUSH_ROWS = 4095;         // 4095 * 2^19 < 2^31
__host__ __device__ constexpr uint64_t lp_fixed_bytes(uint64_t kd, uint64_t k) {
  return (((2 * kd + k) * 4 + 127) & ~127ull) + 2 * LP_ST * 8 + 16;
}
// q = rint(v) for |v| < 2^39 as hi 2^20 + lo (|hi|, |lo| <= 2^19).  hf = v
// rounded to a multiple of 2^20 (adding 1.5 2^43, whose unit in the last
// place is 2^20, and subtracting it back are exact apart from that rounding);
// lf = v - hf is exact (|lf| <= 2^19 on v's own grid); hi = hf / 2^20 and
// lo = rint(lf) are read from the low bits of a sum with 1.5 2^23, whose
// unit in the last place is 1 (ties to even).  hf is an even integer, so
// rint(v) = hf + rint(lf).
__device__ __forceinline__ void lq_split(float v, int& hi, int& lo) {
  const float hf = __fsub_rn(__fadd_rn(v, 0x1.8p43f), 0x1.8p43f);
  const float lf = __fsub_rn(v, hf);
  hi = (int)(__float_as_uint(__fmaf_rn(hf, 0x1p-20f, 0x1.8p23f)) - 0x4B400000u);
  lo = (int)(__float_as_uint(__fadd_rn(lf, 0x1.8p23f)) - 0x4B400000u);
}
__device__ __forceinline__ void red_s32(int* p, int v) { atomicAdd(p, v); }
// barrier 1 among the worker warps only (barrier 0 is __syncthreads)
__device__ __forceinline__ void workers_sync() {
  asm volatile("bar.sync 1, %0;" ::"r"(LP_WORKERS * 32) : "memory");
}

template <bool D64>
__global__ void __launch_bounds__(LS_THREADS, 1) km_local_sum_pipe_kernel(
    const float* __restrict__ x, uint32_t n, uint32_t d, uint32_t k, uint32_t* __restrict__ assign,
    const int* shift, long long* __restrict__ part, unsigned long long* counts, unsigned long long* cnew,
    const uint32_t* chg, uint32_t lim, long long* sums, uint32_t rows, unsigned long long* timeouts, long long polls) {
  pdl_wait();
  if (km_by_changes(chg, lim)) {
    km_apply_changes(x, n, d, k, assign, shift, sums, counts);
    return;
  }
  using namespace pipe;
  extern __shared__ __align__(128) unsigned char lp_sm[];
  const uint64_t kd = (uint64_t)k * d;
  int* HI = reinterpret_cast<int*>(lp_sm);
  int* LO = HI + kd;
  unsigned int* C = reinterpret_cast<unsigned int*>(LO + kd);
  float* xs = reinterpret_cast<float*>(lp_sm + (((2 * kd + k) * 4 + 127) & ~127ull));
  const uint64_t xst = (uint64_t)rows * d;  // floats per stage
  uint32_t* as = reinterpret_cast<uint32_t*>(xs + LP_ST * xst);
  unsigned long long* full = reinterpret_cast<unsigned long long*>(as + LP_ST * rows);
  unsigned long long* empty = full + LP_ST;
  volatile int* err = reinterpret_cast<volatile int*>(empty + LP_ST);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // a CTA's range is a whole number of chunks, so every chunk starts 16-byte aligned
  const uint64_t per = ((((uint64_t)n + gridDim.x - 1) / gridDim.x + rows - 1) / rows) * rows;
  const uint64_t p0 = (uint64_t)blockIdx.x * per;
  const uint64_t p1 = p0 + per < (uint64_t)n ? p0 + per : (uint64_t)n;
  const uint32_t nchunks = p0 < p1 ? (uint32_t)((p1 - p0 + rows - 1) / rows) : 0u;
  const uint32_t fc = rows < LP_FLUSH_ROWS ? LP_FLUSH_ROWS / rows : 1u;  // chunks per window
  for (uint64_t i = threadIdx.x; i < 2 * kd; i += LS_THREADS) HI[i] = 0;
  for (uint32_t i = threadIdx.x; i < k; i += LS_THREADS) C[i] = 0;
  if (threadIdx.x == 0) {
    *err = 0;
    for (int q = 0; q < LP_ST; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], LP_WORKERS);
    }
    fence_mbar_init();
  }
  __syncthreads();
  long long* P = part + (uint64_t)blockIdx.x * kd;
  bool written = false;  // this thread's elements of the CTA's partial hold a window already
  auto flush = [&](uint32_t t0, uint32_t nt) {
    for (uint64_t i = t0; i < kd; i += nt) {
      const long long v = (long long)HI[i] * (1ll << 20) + (long long)LO[i];
      P[i] = written ? P[i] + v : v;
      HI[i] = 0;
      LO[i] = 0;
    }
    written = true;
  };
  uint32_t issued = 0;  // thread 0: chunks whose copies were started
  if (warp == 0) {
    // ----------------------------------------------------------- producer
    if (lane == 0) {
      for (uint32_t c = 0; c < nchunks; ++c) {
        const uint32_t q = c % LP_ST;
        // the stage's previous chunk must be released by every worker, with
        // no error raised (so it landed) before the stage is refilled
        if (c >= (uint32_t)LP_ST && (!mbar_wait(&empty[q], ((c / LP_ST) + 1) & 1u, err, polls) || *err)) break;
        const uint64_t r0 = p0 + (uint64_t)c * rows;
        const uint32_t nr = (uint32_t)(p1 - r0 < rows ? p1 - r0 : rows);
        const uint32_t xb = nr * d * 4, ab = ((nr + 3) & ~3u) * 4;  // ids rounded up to 16 bytes (buffer padding)
        mbar_expect_tx(&full[q], xb + ab);
        bulk_g2s(xs + q * xst, x + r0 * d, xb, &full[q]);
        bulk_g2s(as + q * rows, assign + r0, ab, &full[q]);
        issued = c + 1;
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------- workers
    const float scale = ldexpf(1.f, *shift);
    const uint32_t wk = (uint32_t)warp - 1;
    for (uint32_t c = 0; c < nchunks; ++c) {
      const uint32_t q = c % LP_ST, par = (c / LP_ST) & 1u;
      const bool ok = !*err && mbar_wait(&full[q], par, err, polls);
      if (ok) {
        const uint64_t r0 = p0 + (uint64_t)c * rows;
        const uint32_t nr = (uint32_t)(p1 - r0 < rows ? p1 - r0 : rows);
        const float* X = xs + q * xst;
        const uint32_t* A = as + q * rows;
        if (D64) {
          // lane holds dimensions lane and lane + 32 of row j
          for (uint32_t j = wk; j < nr; j += LP_WORKERS) {
            const uint32_t cl = km_now(A[j], k);
            if (lane == 0) atomicAdd(&C[cl], 1u);
            const float* row = X + j * 64u;
            const uint32_t b = cl * 64u + lane;
            int h0, l0, h1, l1;
            lq_split(row[lane] * scale, h0, l0);
            lq_split(row[lane + 32] * scale, h1, l1);
            red_s32(HI + b, h0);
            red_s32(LO + b, l0);
            red_s32(HI + b + 32, h1);
            red_s32(LO + b + 32, l1);
          }
        } else {
          for (uint32_t j = wk; j < nr; j += LP_WORKERS) {
            const uint32_t cl = km_now(A[j], k);
            if (lane == 0) atomicAdd(&C[cl], 1u);
            const float* row = X + (uint64_t)j * d;
            const uint32_t b = cl * d;
            for (uint32_t dj = lane; dj < d; dj += 32) {
              int h0, l0;
              lq_split(row[dj] * scale, h0, l0);
              red_s32(HI + b + dj, h0);
              red_s32(LO + b + dj, l0);
            }
          }
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[q]);
      if ((c + 1) % fc == 0 && c + 1 < nchunks) {
        workers_sync();
        flush(threadIdx.x - 32, LP_WORKERS * 32);
        workers_sync();
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *err) {
    // a wait gave up somewhere: only the last LP_ST copies the producer
    // issued can still be in flight; let them land before the CTA leaves
    for (uint32_t w = issued > (uint32_t)LP_ST ? issued - LP_ST : 0u; w < issued; ++w)
      mbar_drain(&full[w % LP_ST], (w / LP_ST) & 1u);
    atomicAdd(timeouts, 1ull);
  }
  for (uint64_t i = p0 + threadIdx.x; i < p1; i += LS_THREADS) km_settle_word(assign, i, k);
  // the last window, by the workers with the same element-to-thread mapping
  // as the windows before (each thread's `written` covers its own elements)
  if (warp != 0) flush(threadIdx.x - 32, LP_WORKERS * 32);
  for (uint32_t i = threadIdx.x; i < k; i += LS_THREADS)
    if (C[i]) atomicAdd(cnew + i, (unsigned long long)C[i]);
}

// Update step for D <= 64 with runs sorted per window (Sec. III-E's array
// container, privatised per thread block as above, with the shared-memory
// atomics taken out of the inner loop).  A CTA walks its contiguous range of
// points in windows of win points (8,192 where the shared memory allows,
// else 4,096: fewer windows, fewer sort phases).  For each window it counting-sorts the point
// indices by cluster in shared memory (a histogram, a scan and a scatter of
// 16-bit indices), then every warp takes an equal slice of the sorted order
// and adds its points run by run in registers: lane l reads up to two
// dimensions of each point (D = 64 with 8-byte-aligned points: 2l and
// 2l + 1 with one 8-byte load, so a warp reads the whole 256-byte row;
// otherwise l and l + 32 where below D) and keeps q = rint(x 2^s) = hi 2^20 + lo (lq_split)
// as two 32-bit sums per dimension; when the cluster changes the run is
// added into the CTA's int64 [k][D] sums with one 64-bit shared-memory add
// per dimension.
// A slice holds at most WS_WIN_MAX / WS_WARPS points, so no 32-bit run sum
// can overflow (256 * 2^19 = 2^27).  The CTA stores its sums as its partial and
// adds its counts to the global counts, like km_local_sum_kernel; the sums are
// the same integers in any order.  No wait of any kind: only plain loads and
// block barriers.
constexpr int WS_THREADS = 1024;
constexpr int WS_WARPS = WS_THREADS / 32;
constexpr uint32_t WS_WIN_MAX = 8192;  // points per window (16-bit positions), or half that
constexpr int WS_UNROLL = 8;       // points in flight per warp
__host__ __device__ constexpr uint64_t ws_smem_bytes(uint64_t k, uint64_t d, uint64_t win) {
  return k * d * 8 + 3 * k * 4 + 3 * win * 2;
}
// add a run's split sums of dimensions j0 and (TWO) j1, when below d, into
// cluster c's int64 sums
template <bool TWO>
__device__ __forceinline__ void ws_flush(long long* S, uint32_t c, uint32_t d, uint32_t j0, uint32_t j1, int h0,
                                         int l0, int h1, int l1) {
  unsigned long long* p = reinterpret_cast<unsigned long long*>(S + (uint64_t)c * d);
  if (j0 < d) atomicAdd(p + j0, (unsigned long long)((long long)h0 * (1ll << 20) + (long long)l0));
  if (TWO && j1 < d) atomicAdd(p + j1, (unsigned long long)((long long)h1 * (1ll << 20) + (long long)l1));
}
// Lanes and dimensions by MODE: WS_D64, D = 64 with 8-byte-aligned rows
// (lane l reads dimensions 2l, 2l + 1 with one 8-byte load); WS_D32,
// D <= 32 (lane l dimension l); WS_DANY, D <= 64 (lane l dimensions l and
// l + 32).
enum { WS_D64 = 0, WS_D32 = 1, WS_DANY = 2 };
template <int MODE>
__global__ void __launch_bounds__(WS_THREADS, 1) km_window_sum_kernel(const float* __restrict__ x, uint32_t n,
                                                                      uint32_t d_arg, uint32_t k, uint32_t win,
                                                                      uint32_t* __restrict__ assign,
                                                                      const int* shift, long long* __restrict__ part,
                                                                      unsigned long long* counts,
                                                                      unsigned long long* cnew, const uint32_t* chg, uint32_t lim,
                                                                      long long* sums) {
  const uint32_t d = MODE == WS_D64 ? 64u : d_arg;  // a constant on the 64-wide path
  constexpr bool TWO = MODE != WS_D32;            // two dimensions per lane
  pdl_wait();
  extern __shared__ __align__(16) unsigned char ws_sm[];
  long long* S = reinterpret_cast<long long*>(ws_sm);
  if (km_by_changes(chg, lim)) {
    if (*chg <= n / KM_DELTA_DIRECT) {
      km_apply_changes(x, n, d, k, assign, shift, sums, counts);
      return;
    }
    // many: the clusters that exchange points are few, and the adds to their
    // sums would queue in L2; collected per CTA first
    unsigned long long* dc = reinterpret_cast<unsigned long long*>(S + (uint64_t)k * d);  // [k] count changes
    for (uint64_t i = threadIdx.x; i < (uint64_t)k * (d + 1); i += WS_THREADS) S[i] = 0;
    __syncthreads();
    km_apply_changes(x, n, d, k, assign, shift, S, dc);
    __syncthreads();
    for (uint64_t i = threadIdx.x; i < (uint64_t)k * d; i += WS_THREADS)
      if (S[i]) atomicAdd(reinterpret_cast<unsigned long long*>(sums) + i, (unsigned long long)S[i]);
    for (uint32_t i = threadIdx.x; i < k; i += WS_THREADS)
      if (dc[i]) atomicAdd(counts + i, dc[i]);
    return;
  }
  uint32_t* hc = reinterpret_cast<uint32_t*>(S + (uint64_t)k * d);
  uint32_t* off = hc + k;
  uint32_t* C = off + k;
  uint16_t* wid = reinterpret_cast<uint16_t*>(C + k);
  uint16_t* perm = wid + win;
  uint16_t* pcl = perm + win;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint64_t i = threadIdx.x; i < (uint64_t)k * d; i += WS_THREADS) S[i] = 0;
  for (uint32_t i = threadIdx.x; i < k; i += WS_THREADS) C[i] = 0;
  const uint32_t j0 = MODE == WS_D64 ? 2 * (uint32_t)lane : (uint32_t)lane;
  const uint32_t j1 = MODE == WS_D64 ? j0 + 1 : j0 + 32;
  const uint64_t per = ((uint64_t)n + gridDim.x - 1) / gridDim.x;
  const uint64_t p0 = (uint64_t)blockIdx.x * per;
  const uint64_t p1 = p0 + per < (uint64_t)n ? p0 + per : (uint64_t)n;
  const float scale = ldexpf(1.f, *shift);
  const uint32_t kl = (k + 31) / 32;  // bins per lane in the scan
  for (uint64_t w0 = p0; w0 < p1; w0 += win) {
    const uint32_t nr = (uint32_t)(p1 - w0 < win ? p1 - w0 : win);
    for (uint32_t t = threadIdx.x; t < k; t += WS_THREADS) hc[t] = 0;
    __syncthreads();  // hc cleared; the previous window's sorted order is no longer read
    for (uint32_t r = threadIdx.x; r < nr; r += WS_THREADS) {
      km_settle_word(assign, w0 + r, k);
      const uint32_t c = cluster_of(assign, w0 + r, k);
      wid[r] = (uint16_t)c;
      atomicAdd(&hc[c], 1u);
    }
    __syncthreads();
    if (warp == 0) {
      // exclusive scan of the window's cluster sizes (lane l: bins l kl ..)
      uint32_t tot = 0;
      for (uint32_t j = 0; j < kl; ++j) {
        const uint32_t c = (uint32_t)lane * kl + j;
        if (c < k) tot += hc[c];
      }
      uint32_t incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      uint32_t run = incl - tot;
      for (uint32_t j = 0; j < kl; ++j) {
        const uint32_t c = (uint32_t)lane * kl + j;
        if (c < k) {
          const uint32_t h = hc[c];
          off[c] = run;
          run += h;
          C[c] += h;
        }
      }
    }
    __syncthreads();
    for (uint32_t r = threadIdx.x; r < nr; r += WS_THREADS) {
      const uint32_t c = wid[r];
      const uint32_t pos = atomicAdd(&off[c], 1u);
      perm[pos] = (uint16_t)r;
      pcl[pos] = (uint16_t)c;
    }
    __syncthreads();
    // warp slices of the sorted order; runs summed in registers
    const uint32_t pw = (nr + WS_WARPS - 1) / WS_WARPS;
    const uint32_t q0 = (uint32_t)warp * pw;
    const uint32_t q1 = q0 + pw < nr ? q0 + pw : nr;
    if (q0 < q1) {
      const float* X = x + w0 * d;
      uint32_t cur = pcl[q0];
      int h0 = 0, l0 = 0, h1 = 0, l1 = 0;
      for (uint32_t q = q0; q < q1; q += WS_UNROLL) {
        float2 v[WS_UNROLL];
        uint32_t cl[WS_UNROLL];
#pragma unroll
        for (int u = 0; u < WS_UNROLL; ++u) {
          const uint32_t qq = q + (uint32_t)u;
          const bool ok = qq < q1;
          cl[u] = ok ? pcl[qq] : cur;
          const float* row = X + (uint64_t)(ok ? perm[qq] : 0) * d;
          if (MODE == WS_D64) {
            v[u] = ok ? __ldg(reinterpret_cast<const float2*>(row) + lane) : make_float2(0.f, 0.f);
          } else {
            v[u].x = ok && j0 < d ? __ldg(row + j0) : 0.f;
            v[u].y = TWO && ok && j1 < d ? __ldg(row + j1) : 0.f;
          }
        }
#pragma unroll
        for (int u = 0; u < WS_UNROLL; ++u) {
          if (cl[u] != cur) {  // warp-uniform: the run of cluster cur ended
            ws_flush<TWO>(S, cur, d, j0, j1, h0, l0, h1, l1);
            h0 = l0 = h1 = l1 = 0;
            cur = cl[u];
          }
          int a, b;
          lq_split(v[u].x * scale, a, b);
          h0 += a;
          l0 += b;
          if (TWO) {
            lq_split(v[u].y * scale, a, b);
            h1 += a;
            l1 += b;
          }
        }
      }
      ws_flush<TWO>(S, cur, d, j0, j1, h0, l0, h1, l1);
    }
  }
  __syncthreads();
  long long* P = part + (uint64_t)blockIdx.x * k * d;
  for (uint64_t i = threadIdx.x; i < (uint64_t)k * d; i += WS_THREADS) P[i] = S[i];
  for (uint32_t i = threadIdx.x; i < k; i += WS_THREADS)
    if (C[i]) atomicAdd(cnew + i, (unsigned long long)C[i]);
}

// The centroids of the next round, one CTA per centroid: after a full update
// the sum of the g partials of each dimension becomes the cluster's sum (the
// sorted update and the update by changes left it there), c_k =
// (sum_k * 2^-s) / count_k in FP64, rounded to FP32 (an empty cluster keeps
// c_k), and what the next distance pass and re-check need of them: the shifted
// norm cn[k] = ||c_k - center||^2 (FP32 FMAs; center null: no shift), the
// largest norm, the transposed copy ct, the wide pass's operands bop (null:
// none), each centroid's drift so far and the largest of the round (drift null:
// not kept) and cleared counters.  first: only the
// latter, for the initial centroids.
constexpr uint32_t KM_STATE = 8;  // of the counters: points listed, mode, rounds, length of a rest
__device__ __forceinline__ void km_next_mode(uint32_t* st, uint32_t n);
constexpr int RF_THREADS = 256;
constexpr uint32_t RF_FEW = 8;  // partials
__global__ void __launch_bounds__(RF_THREADS) km_finalize_kernel(const long long* __restrict__ part, uint32_t g,
                                                                 long long* sums, float* c, uint32_t k, uint32_t d,
                                                                 unsigned long long* counts,
                                                                 unsigned long long* cnew,
                                                                 const uint32_t* chg, uint32_t lim, uint32_t* chg_next,
                                                                 const int* shift,
                                                                 const float* __restrict__ center,
                                                                 float* __restrict__ cn, unsigned int* cmax,
                                                                 float* __restrict__ ct, uint8_t* bop,
                                                                 float* drift, unsigned int* maxdrift, uint32_t n,
                                                                 uint32_t* nflag, uint32_t first) {
  pdl_wait();
  __shared__ long long red[RF_THREADS / 32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t kd = (uint64_t)k * d, kk = blockIdx.x, row = kk * d;
  const bool full = !km_by_changes(chg, lim);
  const unsigned long long cnt = first ? 0 : full ? cnew[kk] : counts[kk];
  const double inv = cnt ? ldexp(1.0, -*shift) : 0.0;
  float nrm = 0.f, moved2 = 0.f;
  // Many partials are summed by the warps together, 32 dimensions at a time; with
  // few or none each warp takes 32 dimensions of its own (2,000 x 500, K = 20, two
  // partials, three rounds: 990 us with the warps in step over every 32 dimensions,
  // now 936; 20,000 x 300, K = 64, whose sums lie ready after many rounds, 1,630
  // and 1,511).
  const bool spread = !(full && cnt && part) || g <= RF_FEW;
  __shared__ float tails[2][RF_THREADS / 32];
  __syncthreads();  // every thread has read the count that is cleared below
  for (uint32_t j0 = spread ? 32 * w : 0; j0 < d; j0 += spread ? RF_THREADS : 32) {
    const uint32_t j = j0 + lane;
    long long a = 0;
    if (full && cnt && part && spread) {
      if (j < d)
        for (uint32_t q = 0; q < g; ++q) a += part[(uint64_t)q * kd + row + j];
    } else if (full && cnt && part) {
      if (j < d) {
#pragma unroll 4
        for (uint32_t q = w; q < g; q += RF_THREADS / 32) a += part[(uint64_t)q * kd + row + j];
      }
      __syncthreads();  // the previous dimensions' sums have been read
      red[w][lane] = a;
      __syncthreads();
    }
    if ((spread || w == 0) && j < d) {
      if (full && part) {
        if (cnt && !spread) {
#pragma unroll
          for (int i = 1; i < RF_THREADS / 32; ++i) a += red[i][lane];
        }
        if (!first) sums[row + j] = a;
      } else if (cnt) {
        a = sums[row + j];
      }
      const float was = c[row + j];
      const float v = cnt ? (float)(((double)a * inv) / (double)cnt) : was;
      if (cnt) c[row + j] = v;
      moved2 = fmaf(v - was, v - was, moved2) + (v != was ? 1e-36f : 0.f);  // (tiny squares are flushed)
      ct[(uint64_t)j * k + kk] = v;
      const float t = center ? __fsub_rn(v, center[j]) : v;
      nrm = fmaf(t, t, nrm);
      if (bop) tc::put_operand(bop, d, (uint32_t)kk, j, t);
    }
  }
  if (spread || w == 0) {
    for (int o = 16; o; o >>= 1) {
      nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
      moved2 += __shfl_xor_sync(0xffffffffu, moved2, o);
    }
  }
  if (spread) {
    if (lane == 0) tails[0][w] = nrm, tails[1][w] = moved2;
    __syncthreads();
  }
  if (w == 0) {
    if (lane == 0) {
      for (int i = 1; spread && i < RF_THREADS / 32; ++i) nrm += tails[0][i], moved2 += tails[1][i];
      cn[kk] = nrm;
      if (drift) {
        const float dr = __fmul_ru(__fsqrt_ru(moved2), 1.0001f);  // (the sum's relative error is below 1e-5 at D <= 64)
        drift[kk] = first ? 0.f : __fadd_ru(drift[kk], dr);
        if (!first) atomicMax(maxdrift, __float_as_uint(dr));
      }
      atomicMax(cmax, __float_as_uint(sqrtf(nrm)));
      if (full) counts[kk] = cnt;
      cnew[kk] = 0;
      if (kk == 0) {
        nflag[1] = nflag[4] = 0;  // points to re-check, pairs
        *chg_next = 0;
        if (drift && !first) km_next_mode(nflag + KM_STATE, n);
      }
    }
  }
}

// ------------------------------------------------------------- the filter
// After the first rounds most points cannot change cluster (on a mixture of
// 256 Gaussians in 64 dimensions, K = 256: 82, 75, 40, 25, 15, 14, 13, 11, 12%
// of the points could in rounds 2 to 10), and the triangle inequality tells
// which without computing a distance (Hamerly, "Making k-means even faster",
// 2010): with ub >= the distance to the own centroid a and lb <= the distance
// to every other one, both moved along by the centroids' drifts, the point
// keeps a if ub < lb, or if ub < half the distance from a to the nearest other
// centroid.  Bounds come from the distance and settle passes with their error
// bounds added, are stored relative to the drifts so far (so a skipped point
// writes nothing) and are compared with more slack than all roundings, so a
// skipped point's assignment is the FP64 definition's, by a relative margin of
// 1e-5.  The listed points go through the distance pass by index.
//
// Data without clusters leaves it nothing to skip for many rounds (of normal
// points in 64 dimensions, K = 256, over 99% are listed for six rounds and 93% in
// the tenth; of the mixture's never more than 82%), and a round whose list is not
// used has paid for it.  So the centroids' kernel decides the next round's mode
// (km_next_mode): after two rounds that listed all but 1 / 128 of the points
// the filter rests for three rounds, and no bounds are written; one round then
// writes them again and the next one filters.  After a rest, one round whose
// list is not used (km_use_list) starts another, twice as long.
//
// st: points listed, mode, rounds (that listed nearly all; of the rest, left), length of the last rest.
__device__ __forceinline__ void km_next_mode(uint32_t* st, uint32_t n) {
  const uint32_t listed = st[0];
  uint32_t mode = st[1], rounds = st[2], rest = st[3];
  if (mode == KM_REST) {
    if (--rounds == 0) mode = KM_BOUNDS;
  } else if (mode == KM_BOUNDS) {
    mode = KM_FILTER;
  } else {
    rounds = listed > n - n / 128 ? rounds + 1 : 0;
    if (rest ? !tc::km_use_list(listed, n) : rounds == 2) {
      mode = KM_REST;
      rounds = rest = rest ? min(2 * rest, 1u << 20) : 3;
    }
  }
  st[1] = mode, st[2] = rounds, st[3] = rest;
}

// km_half_kernel: half[k], one CTA per centroid, one thread per other centroid;
// and the largest drift of the round added to the sum of them.
constexpr int HALF_THREADS = 256;
__global__ void __launch_bounds__(HALF_THREADS) km_half_kernel(const float* __restrict__ c,
                                                               const float* __restrict__ ct, uint32_t k, uint32_t d,
                                                               float* __restrict__ half, unsigned int* maxdrift,
                                                               float* far, uint32_t n, uint32_t* nact,
                                                               const uint32_t* mode) {
  pdl_wait();
  __shared__ float own[64], red[HALF_THREADS / 32];
  const uint32_t i = blockIdx.x;
  const bool on = *mode == KM_FILTER;
  if (i == 0 && threadIdx.x == 0) {
    *far = __fadd_ru(*far, __uint_as_float(*maxdrift));
    *maxdrift = 0;
    *nact = on ? 0 : n;
  }
  if (!on) return;
  for (uint32_t t = threadIdx.x; t < d; t += HALF_THREADS) own[t] = c[(uint64_t)i * d + t];
  __syncthreads();
  float best = INFINITY;
  for (uint32_t j = threadIdx.x; j < k; j += HALF_THREADS) {
    float s = 0.f;
#pragma unroll 16
    for (uint32_t t = 0; t < d; ++t) {
      const float v = __ldg(ct + (uint64_t)t * k + j) - own[t];
      s = fmaf(v, v, s);
    }
    if (j != i) best = s != s ? 0.f : fminf(best, s);  // (NaN: no bound; no thread has two centroids at K <= 256)
  }
  for (int o = 16; o; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < HALF_THREADS / 32; ++w) best = fminf(best, red[w]);
    half[i] = 0.5f * __fsqrt_rd(best) * 0.9999f;
  }
}
// Bound by the 12 bytes a point it reads (4M points: 14 us).
constexpr int FI_THREADS = 1024;
__global__ void __launch_bounds__(FI_THREADS) km_filter_kernel(const uint32_t* __restrict__ assign, uint32_t n,
                                                               uint32_t k, KmBounds B, const float* __restrict__ half,
                                                               uint32_t* __restrict__ act, uint32_t* nact) {
  pdl_wait();
  if (*B.mode != KM_FILTER) return;
  __shared__ float s_drift[256], s_half[256];
  __shared__ uint32_t wcnt[FI_THREADS / 32], s_base;
  for (uint32_t i = threadIdx.x; i < k; i += FI_THREADS) s_drift[i] = B.drift[i], s_half[i] = half[i];
  const float far = *B.far;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint64_t b = (uint64_t)blockIdx.x * FI_THREADS * 4; b < n; b += (uint64_t)gridDim.x * FI_THREADS * 4) {
    const uint64_t i0 = b + 4 * threadIdx.x;  // four consecutive points per thread
    uint32_t w[4];
    float u[4], l[4];
    if (i0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(assign + i0);
      const float4 uv = *reinterpret_cast<const float4*>(B.ub + i0), lv = *reinterpret_cast<const float4*>(B.lb + i0);
      w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
      u[0] = uv.x, u[1] = uv.y, u[2] = uv.z, u[3] = uv.w;
      l[0] = lv.x, l[1] = lv.y, l[2] = lv.z, l[3] = lv.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool in = i0 + q < n;
        w[q] = in ? assign[i0 + q] : 0u;
        u[q] = in ? B.ub[i0 + q] : 0.f;
        l[q] = in ? B.lb[i0 + q] : 0.f;
      }
    }
    __syncthreads();  // the drifts are loaded; the previous batch's counts have been read
    uint32_t on = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t a = km_now(w[q], k);
      const float dr = s_drift[a];
      // 2.4e-7: two roundings of each sum
      const float ub = u[q] + dr + 2.4e-7f * (fabsf(u[q]) + dr);
      const float lb = l[q] - far - 2.4e-7f * (fabsf(l[q]) + far);
      if (i0 + q < n && !(ub * 1.00001f < fmaxf(lb, s_half[a]))) on |= 1u << q;
    }
    const uint32_t c = __popc(on);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wcnt[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t t = wcnt[lane];
      uint32_t ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, ti, o);
        if (lane >= o) ti += v;
      }
      wcnt[lane] = ti - t;
      if (lane == 31) s_base = ti ? atomicAdd(nact, ti) : 0u;
    }
    __syncthreads();
    uint32_t at = s_base + wcnt[warp] + incl - c;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (on >> q & 1) act[at++] = (uint32_t)(i0 + q);
  }
}

__global__ void km_finish_kernel(const float* c, uint64_t kd, float* out_c, const uint32_t* assign, uint32_t n,
                                 int32_t* out_a, const unsigned long long* stats, unsigned long long* out_s,
                                 uint32_t iters, volatile uint64_t* host) {
  pdl_wait();
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = tid; i < kd; i += nth) out_c[i] = c[i];
  uint64_t done = 0;
  if (((reinterpret_cast<uintptr_t>(out_a) | reinterpret_cast<uintptr_t>(assign)) & 15) == 0) {
    const uint64_t n4 = n / 4;
    for (uint64_t i = tid; i < n4; i += nth) {
      const uint4 w = reinterpret_cast<const uint4*>(assign)[i];
      reinterpret_cast<uint4*>(out_a)[i] =
          make_uint4(w.x & 0xffffu, w.y & 0xffffu, w.z & 0xffffu, w.w & 0xffffu);
    }
    done = n4 * 4;
  }
  for (uint64_t i = done + tid; i < n; i += nth) out_a[i] = (int32_t)(assign[i] & 0xffffu);
  if (tid == 0) {
    if ((kd + n) & 1) out_a[n] = 0;  // the zero padding before the 8-byte aligned stats
    out_s[0] = stats[0];
    out_s[1] = stats[1];
    out_s[2] = iters;
    out_s[3] = stats[3];
    if (host) *host = stats[3];
  }
}

inline uint64_t a256(uint64_t x) { return (x + 255) & ~255ull; }

}  // namespace

// A job needs no more memory than the form that kept lists of one purpose each
// did, so a budget that held it holds it: the transposed centroids lie in the
// result's place for the centroids, which the last kernel writes; the sorted
// update's cursors and the norms share theirs (the distance pass has read the
// norms by then, and the centroids' kernel makes the next ones after the sums).
size_t km_scratch_bytes(uint32_t n, uint32_t d, uint32_t k, bool wide) {
  uint64_t b = 0;
  b += a256((uint64_t)k * d * 4);      // cent
  b += a256((uint64_t)n * 4 + 16);     // assign (+16: the update copies ids in 16-byte units)
  b += a256((uint64_t)k * d * 8);      // sums
  b += a256((uint64_t)k * 8 * 2);      // counts, counts of a full update
  b += 256;                            // stats, counters (nflag, maxabs, cmax, pairs), shift
  b += a256((uint64_t)n * 4);          // points to re-check; the sorted update's permutation
  b += a256((uint64_t)n * sizeof(KmFew));  // points with a few candidates
  b += a256((uint64_t)k * 4);          // ||c||^2; per-cluster write cursor
  if (wide || km_tc_supported(d, k)) b += a256((uint64_t)d * 4);  // center
  if (local_sums_fit(d, k)) b += a256((uint64_t)LS_MAX_CTAS * k * d * 8);  // per-CTA partial sums
  if (wide) b += a256(km_wide_operand_bytes(d, k));
  return (size_t)b;
}

cudaError_t km_carve(KmBuffers& b, uint8_t* p, size_t bytes, bool wide) {
  const uint64_t n = b.n, d = b.d, k = b.k;
  uint8_t* q = p;
  auto take = [&](uint64_t sz) { uint8_t* r = q; q += a256(sz); return r; };
  b.cent = reinterpret_cast<float*>(take(k * d * 4));
  b.assign = reinterpret_cast<uint32_t*>(take(n * 4 + 16));
  b.sums = reinterpret_cast<long long*>(take(k * d * 8));
  b.counts = reinterpret_cast<unsigned long long*>(take(k * 8 * 2));
  uint8_t* ctl = take(256);
  b.stats = reinterpret_cast<unsigned long long*>(ctl);
  b.nflag = reinterpret_cast<uint32_t*>(ctl + 64);  // 24 words are cleared: to ctl + 160
  b.maxabs = reinterpret_cast<unsigned int*>(b.nflag + 2);
  b.shift = reinterpret_cast<int*>(ctl + 128);
  b.flagged = reinterpret_cast<uint32_t*>(take(n * 4));
  b.pairs = reinterpret_cast<KmFew*>(take(n * sizeof(KmFew)));
  b.cnorm = reinterpret_cast<float*>(take(k * 4));
  b.kcursor = reinterpret_cast<uint32_t*>(b.cnorm);
  b.center = wide || km_tc_supported(b.d, b.k) ? reinterpret_cast<float*>(take(d * 4)) : nullptr;
  b.part = local_sums_fit(d, k) ? reinterpret_cast<long long*>(take((uint64_t)LS_MAX_CTAS * k * d * 8)) : nullptr;
  b.bop = wide ? take(km_wide_operand_bytes((uint32_t)d, (uint32_t)k)) : nullptr;
  if ((uint64_t)(q - p) > bytes) return cudaErrorInvalidValue;
  return cudaSuccess;
}

size_t km_bounds_bytes(uint32_t n, uint32_t k) { return 3 * a256((uint64_t)n * 4) + 2 * a256((uint64_t)k * 4); }

void km_carve_bounds(KmBuffers& b, uint8_t* p) {
  auto take = [&](uint64_t words) { uint8_t* r = p; p += a256(words * 4); return r; };
  b.bounds.ub = reinterpret_cast<float*>(take(b.n));
  b.bounds.lb = reinterpret_cast<float*>(take(b.n));
  b.act = reinterpret_cast<uint32_t*>(take(b.n));
  b.bounds.drift = reinterpret_cast<float*>(take(b.k));
  b.half = reinterpret_cast<float*>(take(b.k));
  b.bounds.far = reinterpret_cast<float*>(b.shift) + 2;
  b.bounds.mode = b.nflag + KM_STATE + 1;
}

// The filter pays for its two kernels (10 - 24 us a round) and the bounds the
// first rounds write for nothing where the distance pass is long enough and
// enough rounds follow: ten, or five if it has 10^8 distances.  Calls with /
// without it, us, of a mixture of 256 Gaussians, and of normal points, which
// leave it little to skip for many rounds (it rests, see km_next_mode; each round
// at rest still costs two launches, and without resting the last column's
// first figures were 2 to 4% higher):
//                                 mixture            normal
//   400K x 8,  K = 40   10 rounds   648 / 656        671 / 674
//   400K x 37, K = 100   5          462 / 435        508 / 471     (left out)
//                        9          686 / 691        840 / 780     (left out)
//                       10          725 / 757        916 / 859
//                       20        1,036 / 1,378    1,668 / 1,613
//   400K x 64, K = 256   5          487 / 525        615 / 574
//                       10          747 / 947      1,130 / 1,060
//   1M x 16,   K = 100   5          734 / 759        839 / 799
//                       10        1,058 / 1,378    1,432 / 1,474
//   1M x 64,   K = 256  10        1,161 / 1,764    2,062 / 1,967
//   4M x 64,   K = 256  10        2,913 / 5,784    6,614 / 6,483
//                       20        4,099 / 11,091  12,285 / 12,404
bool km_bounds_pay(uint32_t n, uint32_t k, uint32_t iters) {
  return n >= 3u << 17 && (iters >= 10 || (iters >= 5 && (uint64_t)n * k >= 100'000'000));
}

cudaError_t launch_kmeans_tc_assign(const float* x, uint32_t n, uint32_t d, const float* c, uint32_t k,
                                    KmBuffers& b, const unsigned int* cmax, uint32_t* nchg, const DevInfo& di,
                                    cudaStream_t s, uint64_t* nk, bool maxabs, const uint32_t* act,
                                    const uint32_t* nact);

cudaError_t launch_kmeans_wide_assign(const float* x, uint32_t n, uint32_t d, uint32_t k, KmBuffers& b,
                                      const unsigned int* cmax, uint32_t* nchg, const DevInfo& di, cudaStream_t s,
                                      uint64_t* nk, bool maxabs);

cudaError_t launch_kmeans(const float* x, const float* init, uint32_t iters, KmBuffers& b, const DevInfo& di,
                          cudaStream_t s, float* out_c, int32_t* out_a, unsigned long long* out_s, uint64_t* nk) {
  cudaError_t e;
  const uint32_t n = b.n, d = b.d, k = b.k;
  int* shift = b.shift;
  float* ct = out_c;  // [d][k] transposed centroids, until km_finish_kernel writes the result there
  auto cmax_of = [&](uint32_t it) { return b.nflag + 6 + (it & 1); };  // max ||c||, one word per parity of the round
  // The distance pass only has to settle the clear cases (every near tie is
  // re-checked), so an FP32 job takes the tensor-core pass on split operands
  // wherever that covers its shape: the assignments are the FP64 definition's
  // either way.  At 200,003 x 37, K = 100 the pass takes 32 us instead of 156
  // and the whole ten-round call 0.69 ms instead of 2.11.  A context that has set
  // a wait limit or stops the copies (diagnostics of the pipelined passes) keeps
  // FP32 jobs on the SIMT pass, which waits on nothing.
  const bool plain = b.polls < 0 && b.stop_copies == 0;
  const bool tc = b.precision != MR_KM_FP32 || (km_tc_supported(d, k) && plain);
  const bool wide = !tc && b.bop && plain;
  const int asm_bytes = (DC_MAX * CS_LD + DC_MAX * XS_LD) * 4;
  if ((e = allow_smem<km_assign_fp32_kernel<true>>(di)) != cudaSuccess ||
      (e = allow_smem<km_assign_fp32_kernel<false>>(di)) != cudaSuccess ||
      (e = allow_smem<km_count_kernel>(di)) != cudaSuccess || (e = allow_smem<km_scatter_kernel>(di)) != cudaSuccess)
    return e;
  const int ls_bytes = (int)((uint64_t)k * d * 8 + (uint64_t)k * 4);
  const bool local = b.part != nullptr && ls_bytes <= di.smem_optin;
  if (local && (e = allow_smem<km_local_sum_kernel>(di)) != cudaSuccess) return e;
  // pipelined update: rows of a multiple of 4 floats, 16-byte aligned points, and a ring of >= 4 rows a stage
  uint32_t lp_rows = 0;
  int lp_bytes = 0;
  if (local && d % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0) {
    const uint64_t fixed = lp_fixed_bytes((uint64_t)k * d, k);
    const uint64_t avail = (uint64_t)di.smem_optin > fixed ? (uint64_t)di.smem_optin - fixed : 0;
    uint64_t r = avail / LP_ST / ((uint64_t)d * 4 + 4);
    if (r > LP_CHUNK_MAX / ((uint64_t)d * 4)) r = LP_CHUNK_MAX / ((uint64_t)d * 4);
    r &= ~3ull;
    if (r >= 4) {
      lp_rows = (uint32_t)r;
      lp_bytes = (int)(fixed + LP_ST * r * ((uint64_t)d * 4 + 4));
      if ((e = allow_smem<km_local_sum_pipe_kernel<true>>(di)) != cudaSuccess ||
          (e = allow_smem<km_local_sum_pipe_kernel<false>>(di)) != cudaSuccess)
        return e;
    }
  }
  // the window-sorted update: D <= 64, sums and window buffers in shared
  // memory (8-byte loads for D = 64 with 8-byte-aligned points)
  const uint32_t ws_win =
      ws_smem_bytes(k, d, WS_WIN_MAX) <= (uint64_t)di.smem_optin ? WS_WIN_MAX : WS_WIN_MAX / 2;
  const bool wsum = local && d <= 64 && ws_smem_bytes(k, d, ws_win) <= (uint64_t)di.smem_optin;
  auto ws_kernel = d == 64 && (reinterpret_cast<uintptr_t>(x) & 7) == 0 ? km_window_sum_kernel<WS_D64>
                   : d <= 32                                               ? km_window_sum_kernel<WS_D32>
                                                                           : km_window_sum_kernel<WS_DANY>;
  if (wsum && ((e = allow_smem<km_window_sum_kernel<WS_D64>>(di)) != cudaSuccess ||
               (e = allow_smem<km_window_sum_kernel<WS_D32>>(di)) != cudaSuccess ||
               (e = allow_smem<km_window_sum_kernel<WS_DANY>>(di)) != cudaSuccess))
    return e;
  uint32_t ls_grid = (uint32_t)di.sms < LS_MAX_CTAS ? (uint32_t)di.sms : LS_MAX_CTAS;
  if ((uint64_t)ls_grid * 1024 > n) ls_grid = (uint32_t)((n + 1023) / 1024);
  if (b.grid_cap && ls_grid > b.grid_cap) ls_grid = b.grid_cap;
  if (ls_grid < 1) ls_grid = 1;
  const long long polls = b.polls < 0 ? pipe::SPIN_LIMIT : b.polls;
  const int set_t = set_threads(k);
  const size_t set_bytes = set_smem(d, k);
  auto set_kernel = k > (uint32_t)set_t ? km_settle_kernel<true> : km_settle_kernel<false>;
  if ((e = allow_smem<km_settle_kernel<true>>(di)) != cudaSuccess ||
      (e = allow_smem<km_settle_kernel<false>>(di)) != cudaSuccess)
    return e;
  const uint32_t ntiles = (n + TP - 1) / TP;
  uint32_t agrid = ntiles < (uint32_t)di.sms * 2 ? ntiles : (uint32_t)di.sms * 2;
  if (b.grid_cap && agrid > b.grid_cap) agrid = b.grid_cap;
  km_setup_kernel<<<(d + 31) / 32, SETUP_THREADS, 0, s>>>(init, k, d, b.cent, b.center, b.counts + k, b.nflag,
                                                          b.stats);
  ++*nk;
  // the fixed-point scale needs max |x|: a pass of its own for the SIMT
  // path; the tensor-core pass finds it while converting the first iteration
  if (!tc && !wide) {
    km_maxabs_kernel<<<di.sms * 4, 256, 0, s>>>(x, (uint64_t)n * d, b.maxabs);
    ++*nk;
  }
  // rows and dimensions past K and D stay zero
  if (wide && (e = cudaMemsetAsync(b.bop, 0, km_wide_operand_bytes(d, k), s)) != cudaSuccess) return e;
  const bool filter = tc && b.bounds.ub;
  float* drift = filter ? const_cast<float*>(b.bounds.drift) : nullptr;
  unsigned int* maxdrift = reinterpret_cast<unsigned int*>(shift) + 1;
  float* far = reinterpret_cast<float*>(shift) + 2;
  uint32_t* nact = b.nflag + KM_STATE;
  const KmBounds bounds = filter ? b.bounds : KmBounds{};
  const float* center = tc || wide ? b.center : nullptr;
  const uint32_t lim = n / (wsum ? KM_DELTA_WINDOW : local ? KM_DELTA_LOCAL : KM_DELTA_SORTED);  // points moved, at most, in an update by changes
  auto chg_of = [&](uint32_t it) { return b.nflag + ((it & 1) ? 5 : 0); };  // points that changed cluster in the round
  auto finalize = [&](uint32_t it, bool first) {
    ++*nk;
    return launch_pdl(km_finalize_kernel, dim3(k), dim3(RF_THREADS), 0, s,
                      local ? (const long long*)b.part : (const long long*)nullptr, ls_grid, b.sums, b.cent, k, d,
                      b.counts, b.counts + k, it > 1 ? (const uint32_t*)chg_of(it - 1) : (const uint32_t*)nullptr, lim,
                      chg_of(it),
                      (const int*)shift, center, b.cnorm, cmax_of(it), ct, wide ? b.bop : (uint8_t*)nullptr, drift,
                      maxdrift, n, b.nflag, first ? 1u : 0u);
  };
  if ((e = finalize(0, true)) != cudaSuccess) return e;
  unsigned long long* cnew = b.counts + k;
  for (uint32_t it = 0; it < iters; ++it) {
    uint32_t* chg = it ? chg_of(it) : nullptr;
    // kernels that follow another kernel of this job on the stream start
    // while it drains (programmatic dependent launch; each waits first)
    if (tc) {
      const bool skip = filter && it > 0;
      if (skip) {
        const uint64_t fb = ((uint64_t)n + FI_THREADS * 4 - 1) / (FI_THREADS * 4);
        if ((e = launch_pdl(km_half_kernel, dim3(k), dim3(HALF_THREADS), 0, s, (const float*)b.cent,
                            (const float*)ct, k, d, b.half, maxdrift, far, n, nact, bounds.mode)) != cudaSuccess ||
            (e = launch_pdl(km_filter_kernel, dim3((unsigned)(fb < 2ull * di.sms ? fb : 2ull * di.sms)),
                            dim3(FI_THREADS), 0, s, (const uint32_t*)b.assign, n, k, bounds, (const float*)b.half,
                            b.act, nact)) != cudaSuccess)
          return e;
        *nk += 2;
      }
      if ((e = launch_kmeans_tc_assign(x, n, d, b.cent, k, b, cmax_of(it), chg, di, s, nk, it == 0,
                                       skip ? b.act : nullptr, nact)) != cudaSuccess)
        return e;
    } else if (wide) {
      if ((e = launch_kmeans_wide_assign(x, n, d, k, b, cmax_of(it), chg, di, s, nk, it == 0)) != cudaSuccess)
        return e;
    } else {
      if ((e = kt_begin(b.kt, s)) != cudaSuccess) return e;
      (k <= 256 ? km_assign_fp32_kernel<true> : km_assign_fp32_kernel<false>)<<<agrid, KM_THREADS, asm_bytes, s>>>(
          x, n, d, b.cent, k, b.cnorm, cmax_of(it), b.assign, chg, b.flagged, b.nflag + 1, b.pairs, b.nflag + 4);
      if ((e = cudaGetLastError()) != cudaSuccess || (e = kt_end(b.kt, s)) != cudaSuccess) return e;
      ++*nk;
    }
    if ((e = launch_pdl(set_kernel, dim3(di.sms * (2048 / set_t < 8 ? 2048 / set_t : 8)), dim3(set_t), set_bytes, s, x,
                        n, d, (const float*)b.cent, (const float*)ct, k, (const KmFew*)b.pairs,
                        (const uint32_t*)(b.nflag + 4), (const uint32_t*)b.flagged, (const uint32_t*)(b.nflag + 1),
                        b.assign, chg, b.stats, it == 0 ? (const unsigned int*)b.maxabs : (const unsigned int*)nullptr,
                        shift, cmax_of(it + 1), bounds)) != cudaSuccess)
      return e;
    ++*nk;
    if (local) {  // update with local arrays
      if (wsum)
        e = launch_pdl(ws_kernel, dim3(ls_grid),
                       dim3(WS_THREADS), (size_t)ws_smem_bytes(k, d, ws_win), s, x, n, d, k, ws_win,
                       b.assign, (const int*)shift, b.part, b.counts, cnew, (const uint32_t*)chg, lim, b.sums);
      else if (lp_rows)
        e = launch_pdl(d == 64 ? km_local_sum_pipe_kernel<true> : km_local_sum_pipe_kernel<false>, dim3(ls_grid),
                       dim3(LS_THREADS), (size_t)lp_bytes, s, x, n, d, k, b.assign, (const int*)shift,
                       b.part, b.counts, cnew, (const uint32_t*)chg, lim, b.sums, lp_rows, b.stats + 3, polls);
      else
        e = launch_pdl(km_local_sum_kernel, dim3(ls_grid), dim3(LS_THREADS), (size_t)ls_bytes, s, x, n, d, k,
                       b.assign, (const int*)shift, b.part, b.counts, cnew, (const uint32_t*)chg, lim, b.sums);
      if (e != cudaSuccess) return e;
      ++*nk;
      if ((e = finalize(it + 1, false)) != cudaSuccess) return e;
      continue;
    }
    // update: counting sort of the points by cluster, then run-wise sums
    const uint64_t sc_blocks = (n + (uint64_t)SCAT_THREADS * SCAT_PER_THREAD - 1) / ((uint64_t)SCAT_THREADS * SCAT_PER_THREAD);
    const uint64_t sum_warps = (n + SUM_RUN - 1) / SUM_RUN;
    if ((e = launch_pdl(km_count_kernel, dim3(di.sms * 2), dim3(512), (size_t)k * 4, s, x, d, b.assign, n, k, b.counts,
                        cnew, (const uint32_t*)chg, lim, (const int*)shift, b.sums)) != cudaSuccess ||
        (e = launch_pdl(km_offsets_kernel, dim3(1), dim3(1024), 0, s, (const unsigned long long*)cnew, k, b.kcursor,
                        (const uint32_t*)chg, lim)) != cudaSuccess ||
        (e = launch_pdl(km_scatter_kernel, dim3((unsigned)sc_blocks), dim3(SCAT_THREADS), (size_t)k * 4, s,
                        (const uint32_t*)b.assign, n, k, b.kcursor, b.flagged, (const uint32_t*)chg, lim)) != cudaSuccess ||
        // after the scatter, kcursor[c] is one past the last position of cluster c
        (e = launch_pdl(km_sum_kernel, dim3((unsigned)((sum_warps * 32 + 255) / 256)), dim3(256), 0, s, x, n, d, k,
                        (const uint32_t*)b.kcursor, (const uint32_t*)b.flagged, (const int*)shift, b.sums,
                        (const uint32_t*)chg, lim)) != cudaSuccess)
      return e;
    *nk += 4;  // count, offsets, scatter, sums
    if ((e = cudaGetLastError()) != cudaSuccess || (e = finalize(it + 1, false)) != cudaSuccess) return e;
  }
  if ((e = launch_pdl(km_finish_kernel, dim3(di.sms * 4), dim3(256), 0, s, (const float*)b.cent, (uint64_t)k * d,
                      out_c, (const uint32_t*)b.assign, n, out_a, (const unsigned long long*)b.stats, out_s, iters,
                      (volatile uint64_t*)b.host)) !=
      cudaSuccess)
    return e;
  ++*nk;
  return cudaGetLastError();
}

}  // namespace mrgb
