// Array-container jobs whose key range is large: the 16M-key histogram and
// the k-mer Bloom-filter build (the two applications the paper runs with
// "eliminating local arrays", Sec. III-E and the data-set table of Sec. IV).
//
// Large-key histogram.  Keys are u32; key k < nbins adds one to bin k, any
// other key to bin nbins.  Two containers:
//   * local arrays: one u32 copy of all bins per CTA in shared memory
//     (red.shared), flushed with one global atomic per non-zero bin.  Only
//     possible while nbins + 1 counters fit the opt-in shared memory.
//   * global array (the paper's choice for large arrays): every key is one
//     red.global.add on a single counter array.  While the input has fewer
//     than 2^32 keys the counters are u32, so 16M bins take 64 MiB and stay
//     resident in the 129 MB L2 (the GPU counterpart of the paper's coherent
//     L2 argument); a final pass widens them to the u64 result.
//   Warps combine equal keys first (match.any), which turns the hot keys of
//   a skewed input into one atomic per warp; a warp that sees no repeats over
//   a window of tiles switches the step off and re-probes later.
//
// Bloom-filter build.  Element = every window of L bases of an ASCII DNA
// sequence whose bytes are all A/C/G/T; code = base-4 number of the window,
// first base most significant.  a = mix(code) mod m, b = 1 + mix(code ^
// 0x9E3779B97F4A7C15) mod (m - 1), mix = SplitMix64's output function
// (Steele, Lea & Flood, 2014); bits (a + i b) mod m, i < h, are set with
// atomicOr on u32 words (bit j = bit j%8 of byte j/8 of the result).
// A CTA packs its tile of bases into 2-bit codes (and a 1-bit invalid mask)
// in shared memory, big-endian within each word, so any window's code is one
// 128-bit funnel shift; both reductions mod m use Barrett's method with a
// 64-bit reciprocal computed on the host.
#include "mr_internal.h"

namespace mrgb {
namespace {

constexpr int HK_THREADS = 256;        // global-array kernel
constexpr int HK_SMEM_THREADS = 1024;  // local-array kernel
constexpr int HK_WINDOW = 16;          // tiles per aggregation decision

__device__ __forceinline__ uint4 ldg_nc(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// L2 policies: the streamed keys are marked evict-first and the counters
// evict-last, so the counter array (64 MiB at 16M bins) stays resident in L2
// instead of being written back and re-read as the input streams through.
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint4 ldg_stream_hint(const uint4* p, uint64_t pol) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p), "l"(pol));
  return r;
}

__device__ __forceinline__ void red_add(uint32_t* p, uint32_t v) { atomicAdd(p, v); }
__device__ __forceinline__ void red_add(unsigned long long* p, uint32_t v) { atomicAdd(p, (unsigned long long)v); }
__device__ __forceinline__ void red_add_hint(uint32_t* p, uint32_t v, uint64_t pol) {
  asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void red_add_hint(unsigned long long* p, uint32_t v, uint64_t pol) {
  asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(p), "l"((unsigned long long)v),
               "l"(pol)
               : "memory");
}

__device__ __forceinline__ uint32_t key_at(const uint4& w, int e) {
  return e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w;
}

// Keys are read as 16-byte groups from the 16-byte-aligned address at or
// below the input; group g holds keys 4g - off .. 4g - off + 3 (off = the
// input's misalignment in keys), and keys outside [0, n) are masked.  A group
// that holds at least one key lies in the same aligned 16 bytes as that key,
// so no read leaves the pages of the input.
// One warp of nwarps.
template <typename C>
__device__ __forceinline__ void hk_global_warp(const uint4* __restrict__ base, uint32_t off, uint64_t n, uint32_t nbins,
                                               C* __restrict__ cnt, uint64_t warp, uint64_t nwarps) {
  const int lane = threadIdx.x & 31;
  const uint64_t groups = (n + off + 3) / 4;
  const uint64_t tiles = (groups + 31) / 32;  // one group per lane
  bool agg = true;
  uint32_t saved = 0, win = 0, off_windows = 0;
  const uint64_t pol_in = l2_policy_evict_first(), pol_cnt = l2_policy_evict_last();
  for (uint64_t t = warp; t < tiles; t += nwarps) {
    const uint64_t g = t * 32 + lane;
    uint4 w = make_uint4(0, 0, 0, 0);
    if (g < groups) w = ldg_stream_hint(base + g, pol_in);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t idx = (int64_t)(4 * g + e) - (int64_t)off;
      const bool valid = g < groups && idx >= 0 && (uint64_t)idx < n;
      const uint32_t key = key_at(w, e);
      const uint32_t k = key < nbins ? key : nbins;
      if (agg) {
        const uint32_t vm = __ballot_sync(0xffffffffu, valid);
        const uint32_t m = __match_any_sync(0xffffffffu, k) & vm;
        if (valid && (__ffs(m) - 1) == lane) {
          red_add_hint(cnt + k, (uint32_t)__popc(m), pol_cnt);
          saved += (uint32_t)__popc(m) - 1;
        }
      } else if (valid) {
        red_add_hint(cnt + k, 1u, pol_cnt);
      }
    }
    if (++win == HK_WINDOW) {
      win = 0;
      if (agg) {
        // keep combining while it saves at least 1 atomic in 16
        const uint32_t s = __reduce_add_sync(0xffffffffu, saved);
        agg = s * 16u >= (uint32_t)(HK_WINDOW * 32 * 4);
        saved = 0;
      } else if (++off_windows == 16) {
        off_windows = 0;
        agg = true;  // re-probe: the key mix may have changed
      }
    }
  }
}

template <typename C>
__global__ void __launch_bounds__(HK_THREADS)
hk_global_kernel(const uint4* __restrict__ base, uint32_t off, uint64_t n, uint32_t nbins, C* __restrict__ cnt) {
  hk_global_warp(base, off, n, nbins, cnt, ((uint64_t)blockIdx.x * HK_THREADS + threadIdx.x) >> 5,
                 ((uint64_t)gridDim.x * HK_THREADS) >> 5);
}

// Local arrays: nbins + 1 u32 counters per CTA in shared memory, added straight
// to the u64 result (few enough bins that a u32 array to widen would only add a
// launch).
__global__ void __launch_bounds__(HK_SMEM_THREADS)
hk_smem_kernel(const uint4* __restrict__ base, uint32_t off, uint64_t n, uint32_t nbins,
               unsigned long long* __restrict__ cnt) {
  extern __shared__ uint32_t sh_bins[];
  for (uint32_t i = threadIdx.x; i <= nbins; i += blockDim.x) sh_bins[i] = 0;
  __syncthreads();
  const uint64_t groups = (n + off + 3) / 4;
  for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 w = ldg_nc(base + g);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t idx = (int64_t)(4 * g + e) - (int64_t)off;
      if (idx >= 0 && (uint64_t)idx < n) {
        const uint32_t key = key_at(w, e);
        atomicAdd(&sh_bins[key < nbins ? key : nbins], 1u);
      }
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i <= nbins; i += blockDim.x) {
    const uint32_t v = sh_bins[i];
    if (v) red_add(cnt + i, v);
  }
}

// Local arrays spread over a thread-block cluster: the bins are cut into
// HKC slices of `slice` counters, CTA r of a cluster holding slice r in its
// shared memory, so a cluster holds HKC times as many bins as one CTA (the
// paper's local arrays, Sec. III-E, with a cluster of CTAs as the worker).
// Every CTA streams its share of the keys and adds each one to its slice's
// owner through distributed shared memory (red.shared::cluster); a cluster
// barrier before the first add (every slice zeroed) and after the last (every
// add landed), then each CTA adds its slice's non-zero counters to the global
// array.  No CTA touches another's shared memory after the second barrier,
// so CTAs may then exit in any order.
constexpr int HKC = 8;  // CTAs per cluster (the portable maximum)

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

template <typename C>
__global__ void __launch_bounds__(HK_SMEM_THREADS)
hk_cluster_kernel(const uint4* __restrict__ base, uint32_t off, uint64_t n, uint32_t nbins, uint32_t slice,
                  uint32_t slice_mul, C* __restrict__ cnt) {
  extern __shared__ uint32_t sh_bins[];
  const uint32_t rank = cluster_rank();
  for (uint32_t i = threadIdx.x; i < slice; i += blockDim.x) sh_bins[i] = 0;
  cluster_sync_all();
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sh_bins);
  const uint64_t groups = (n + off + 3) / 4;
  for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 w = ldg_nc(base + g);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t idx = (int64_t)(4 * g + e) - (int64_t)off;
      if (idx >= 0 && (uint64_t)idx < n) {
        const uint32_t key = key_at(w, e);
        const uint32_t k = key < nbins ? key : nbins;
        // owner = k / slice: the multiply-high estimate is at most one low
        uint32_t r = __umulhi(k, slice_mul);
        uint32_t loc = k - r * slice;
        if (loc >= slice) {
          ++r;
          loc -= slice;
        }
        uint32_t ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(sbase + 4 * loc), "r"(r));
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], 1;" ::"r"(ra) : "memory");
      }
    }
  }
  cluster_sync_all();
  const uint64_t b0 = (uint64_t)rank * slice;
  for (uint32_t i = threadIdx.x; i < slice && b0 + i <= nbins; i += blockDim.x) {
    const uint32_t v = sh_bins[i];
    if (v) red_add(cnt + b0 + i, v);
  }
}

__global__ void hk_widen_kernel(const uint32_t* __restrict__ c32, uint64_t nb, unsigned long long* __restrict__ out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = c32[i];
}

// ------------------------------------------------------ partitioned counting
// Bins that do not fit one CTA's shared memory, many keys.  The global-array
// kernel is bound by the L2's atomic rate (about 190G/s: 1.40 ms for 256M
// uniform keys over 16M bins, 12% of the HBM rate), while adds in shared
// memory run several times faster, so the keys are first grouped by ranges of
// 2^PS bins ("ranges"), each of which does fit one CTA:
//   0. hk_look_kernel looks at some of the keys and sends such as sorted ones over
//      few bins to the global array after all.
//   1. hk_part_kernel: a CTA takes chunks of PCHUNK consecutive keys, counts
//      them by bucket (up to 1,024 buckets of 2^F bins, whatever the number of
//      ranges, so that few ranges do not mean few counters and many conflicts)
//      in shared memory, scans the counts into cursors, reads the keys again
//      (they are still in L2; holding them in registers halves the warps an SM
//      runs), places every key at its bucket's cursor and writes the chunk,
//      grouped, as 16-bit offsets within the range.  Where each range starts
//      in the chunk goes into a table [range][chunk].  Bound by the shared
//      memory pipe: three random accesses a key, 3.4 wavefronts per warp each.
//   2. hk_plan_kernel cuts the ranges into units: one, or several over equal
//      parts of the chunks (or of the keys, where those lie in lumps) for a range
//      that holds much more than its share (skewed keys, or few ranges).
//   3. hk_count_kernel: one CTA per unit adds its range's pieces of all chunks
//      into shared memory and stores the counts (u64, no clearing, no widening)
//      or, for a range of several units, adds the non-zero ones.
// HBM traffic: 4 + 2 + 2 bytes a key instead of 4, but no atomics beyond the
// SM: 256M keys over 16M bins take 0.87 ms instead of 1.51 in
// all, skewed ones (rank density 1 / (rank + 1)) 0.87 instead of 8.2.
// A warp whose 128 keys of a load share a bucket (sorted input) moves the cursor
// once.
constexpr int PT = 1024;                // threads of the partition kernel (two CTAs per SM)
constexpr int PV = 8;                   // 16-byte loads per thread and chunk
constexpr int PAHEAD = 2;               // of them in flight
constexpr uint32_t PCHUNK = PT * PV * 4;  // 32,768 keys
constexpr uint32_t PGROUP = 8;          // chunks per 16-byte table write
constexpr uint32_t PS = 15;             // log2 of a range's bins (128 KiB of u32 counters)
constexpr uint32_t PNF = 1024;          // buckets, at most
constexpr uint32_t PRANGES = 1024;      // ranges, at most
constexpr int PCT = 1024;               // threads of the counting kernel
constexpr uint32_t PUNIT_MIN = 1u << 18;  // keys worth a unit of their own (8 per bin)
constexpr uint32_t PUNITS = 256;        // units of an even split

struct PartArgs {
  void* item;          // [chunks][items of a chunk] grouped offsets within the range
  uint16_t* start;     // [ranges + 1][chunks] first item of each range in each chunk
  uint32_t* total;     // [ranges] keys of each range
  uint32_t* most;      // [ranges] its longest piece of a chunk
  uint32_t* cursor;    // [0] the counting kernel's cursor, [1] number of units, [2] the keys take the global array
  uint4* unit;         // {range, first chunk, end chunk, UNIT_* and log2 of a piece's parts << 8}
  uint32_t chunks;     // a multiple of PGROUP
  uint32_t ranges, nf, fshift;
  uint32_t step;       // log2 of the buckets per range
};
constexpr uint32_t UNIT_SEVERAL = 1;  // one of several units of its range, which add to the result
constexpr uint32_t UNIT_LUMPS = 2;    // its keys lie in few of its chunks (sorted keys)

// Exclusive scan in place of nf <= T counters by T threads (entry nf: the total).
template <int T>
__device__ __forceinline__ void block_scan(uint32_t* cnt, uint32_t nf, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t a = threadIdx.x < nf ? cnt[threadIdx.x] : 0;
  uint32_t incl = a;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < T / 32 ? wsum[lane] : 0, wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += v;
    }
    wsum[lane] = wi - w;
    if (lane == 31) cnt[nf] = wi;
  }
  __syncthreads();
  if (threadIdx.x < nf) cnt[threadIdx.x] = wsum[warp] + incl - a;
  __syncthreads();
}

// Chunk c of this CTA's chunks c0 .. c1 - 1 is done: write the starts of the
// chunks since the last write, a whole group at a time where it is this CTA's.
__device__ __forceinline__ void write_starts(const PartArgs& P, const uint16_t* stage, uint32_t c, uint32_t c0,
                                             uint32_t c1) {
  if (c % PGROUP != PGROUP - 1 && c + 1 != c1) return;
  const uint32_t g0 = c / PGROUP * PGROUP;
  for (uint32_t b = threadIdx.x; b <= P.ranges; b += blockDim.x) {
    uint16_t* t = P.start + (uint64_t)b * P.chunks + g0;
    if (g0 >= c0 && c % PGROUP == PGROUP - 1)
      *reinterpret_cast<uint4*>(t) = *reinterpret_cast<const uint4*>(stage + b * PGROUP);
    else
      for (uint32_t q = g0 < c0 ? c0 - g0 : 0; q <= c % PGROUP; ++q) t[q] = stage[b * PGROUP + q];
  }
}
// The scanned bucket counts of chunk c: where its ranges start, their totals and
// (MOST) longest pieces ([ranges] each; hashed bit positions lie in no lumps).
template <bool MOST>
__device__ __forceinline__ void stage_starts(const PartArgs& P, const uint32_t* cnt, uint16_t* stage, uint32_t* tot,
                                             uint32_t c) {
  for (uint32_t b = threadIdx.x; b <= P.ranges; b += blockDim.x) {
    const uint32_t at = cnt[min(b << P.step, P.nf)];
    stage[b * PGROUP + c % PGROUP] = (uint16_t)at;
    if (b < P.ranges) {
      const uint32_t len = cnt[min((b + 1) << P.step, P.nf)] - at;
      tot[b] += len;
      if (MOST) tot[P.ranges + b] = max(tot[P.ranges + b], len);
    }
  }
}
template <bool MOST>
__device__ __forceinline__ void add_totals(const PartArgs& P, const uint32_t* tot) {
  for (uint32_t b = threadIdx.x; b < P.ranges; b += blockDim.x)
    if (tot[b]) {
      atomicAdd(P.total + b, tot[b]);
      if (MOST) atomicMax(P.most + b, tot[P.ranges + b]);
    }
}

// Whether grouping pays is for the keys to say.  Sorted keys over few enough bins
// repeat within a warp's load, and the global-array kernel, which adds equal keys
// of a warp at once, then reads them little slower than memory gives them: 256M
// sorted keys over 1M bins take 0.33 ms there and 0.68 grouped, 16M over 60,000
// 0.048 and 0.165.  So 64
// groups of 128 consecutive keys are looked at (every CTA the same ones): where
// they have at most 16 runs of equal keys on average, and at least half of them
// start with another key than the one before (one hot key would queue at its
// bin), the result is cleared and the keys take the global array.  This kernel
// also clears the totals, for which there was a memory operation.
constexpr int LOOK_T = 1024;
constexpr uint32_t LOOKS = 64, LOOK_RUNS = 16, LOOK_KEYS = 32;
__global__ void __launch_bounds__(LOOK_T) hk_look_kernel(const uint4* __restrict__ base, uint64_t n, PartArgs P,
                                                         uint64_t words, uint32_t add, unsigned long long* __restrict__ out) {
  __shared__ uint32_t s_first[LOOKS], s_runs;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int PER = LOOKS / (LOOK_T / 32);
  const uint64_t tiles = n / 128;  // (a later round of a long input may have none: grouped)
  if (threadIdx.x == 0) s_runs = 0;
  __syncthreads();
  uint4 v[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q)
    v[q] = tiles ? __ldg(base + (PER * warp + q) * tiles / LOOKS * 32 + lane) : make_uint4(0, 1, 2, 3);
  uint32_t runs = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const uint32_t prev = __shfl_up_sync(0xffffffffu, v[q].w, 1);
    runs += (lane == 0 || v[q].x != prev) + (v[q].y != v[q].x) + (v[q].z != v[q].y) + (v[q].w != v[q].z);
    if (lane == 0) s_first[PER * warp + q] = v[q].x;
  }
  runs = __reduce_add_sync(0xffffffffu, runs);
  if (lane == 0) atomicAdd(&s_runs, runs);
  __syncthreads();
  const bool other = threadIdx.x && threadIdx.x < LOOKS && s_first[threadIdx.x] != s_first[threadIdx.x - 1];
  const bool direct = __syncthreads_count(other) >= (int)LOOK_KEYS && s_runs <= LOOK_RUNS * LOOKS;
  if (blockIdx.x == 0) {
    for (uint32_t i = threadIdx.x; i < 2 * P.ranges + 2; i += LOOK_T) P.total[i] = 0;
    if (threadIdx.x == 0) P.cursor[2] = direct;
  }
  if (direct && !add)
    for (uint64_t i = (uint64_t)blockIdx.x * LOOK_T + threadIdx.x; i < words; i += (uint64_t)gridDim.x * LOOK_T) out[i] = 0;
}

__global__ void __launch_bounds__(PT, 2) hk_part_kernel(const uint4* __restrict__ base, uint32_t off, uint64_t n,
                                                        uint32_t nbins, PartArgs P, unsigned long long* __restrict__ result) {
  pdl_wait();
  if (P.cursor[2]) {
    hk_global_warp(base, off, n, nbins, result, ((uint64_t)blockIdx.x * PT + threadIdx.x) >> 5,
                   ((uint64_t)gridDim.x * PT) >> 5);
    return;
  }
  extern __shared__ __align__(16) unsigned char hp_sm[];
  uint16_t* buf = reinterpret_cast<uint16_t*>(hp_sm);                 // [PCHUNK]
  uint32_t* cnt = reinterpret_cast<uint32_t*>(buf + PCHUNK);          // [PNF + 1]
  uint32_t* tot = cnt + PNF + 4;                                      // [2][ranges]
  uint16_t* stage = reinterpret_cast<uint16_t*>(tot + 2 * PRANGES);   // [ranges + 1][PGROUP]
  __shared__ uint32_t wsum[32];
  const int lane = threadIdx.x & 31;
  const uint64_t end = n + off;  // items in group space: item i of the stream is key i - off
  const uint32_t fs = P.fshift;
  for (uint32_t i = threadIdx.x; i < 2 * P.ranges; i += PT) tot[i] = 0;
  const uint32_t per = (P.chunks + gridDim.x - 1) / gridDim.x;
  const uint32_t c0 = blockIdx.x * per, c1 = min(c0 + per, P.chunks);
  for (uint32_t c = c0; c < c1; ++c) {
    const uint64_t i0 = (uint64_t)c * PCHUNK;
    for (uint32_t i = threadIdx.x; i < P.nf; i += PT) cnt[i] = 0;
    __syncthreads();
    const bool whole = i0 >= off && i0 + PCHUNK <= end;  // every item is a key
    const uint4* src = base + i0 / 4 + threadIdx.x;
    if (whole) {
#pragma unroll 1
      for (int q = 0; q < PV; q += PAHEAD) {
        uint4 v[PAHEAD];
#pragma unroll
        for (int t = 0; t < PAHEAD; ++t) v[t] = __ldg(src + (q + t) * PT);
#pragma unroll
        for (int t = 0; t < PAHEAD; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) atomicAdd(cnt + (min(key_at(v[t], e), nbins) >> fs), 1u);
      }
    } else {
      for (int q = 0; q < PV; ++q) {
        const uint64_t e0 = i0 + 4 * ((uint64_t)q * PT + threadIdx.x);
        if (e0 >= end) continue;
        const uint4 v = __ldg(src + q * PT);
        for (int e = 0; e < 4; ++e)
          if (e0 + e >= off && e0 + e < end) atomicAdd(cnt + (min(key_at(v, e), nbins) >> fs), 1u);
      }
    }
    __syncthreads();
    block_scan<PT>(cnt, P.nf, wsum);
    stage_starts<true>(P, cnt, stage, tot, c);
    __syncthreads();  // the starts are read; the counters become cursors
    if (whole) {
#pragma unroll 1
      for (int q = 0; q < PV; q += PAHEAD) {
        uint4 v[PAHEAD];
#pragma unroll
        for (int t = 0; t < PAHEAD; ++t) v[t] = __ldg(src + (q + t) * PT);
#pragma unroll
        for (int t = 0; t < PAHEAD; ++t) {
          uint32_t k[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) k[e] = min(key_at(v[t], e), nbins);
          const uint32_t fw = __shfl_sync(0xffffffffu, k[0] >> fs, 0);
          const uint32_t other = ((k[0] >> fs) ^ fw) | ((k[1] >> fs) ^ fw) | ((k[2] >> fs) ^ fw) | ((k[3] >> fs) ^ fw);
          uint32_t r[4];
          if (__all_sync(0xffffffffu, other == 0)) {
            uint32_t r0 = 0;
            if (lane == 0) r0 = atomicAdd(cnt + fw, 128u);
            r0 = __shfl_sync(0xffffffffu, r0, 0) + 4 * lane;
#pragma unroll
            for (int e = 0; e < 4; ++e) r[e] = r0 + e;
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) r[e] = atomicAdd(cnt + (k[e] >> fs), 1u);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) buf[r[e]] = (uint16_t)(k[e] & ((1u << PS) - 1));
        }
      }
    } else {
      for (int q = 0; q < PV; ++q) {
        const uint64_t e0 = i0 + 4 * ((uint64_t)q * PT + threadIdx.x);
        if (e0 >= end) continue;
        const uint4 v = __ldg(src + q * PT);
        for (int e = 0; e < 4; ++e) {
          const uint32_t k = min(key_at(v, e), nbins);
          if (e0 + e >= off && e0 + e < end) buf[atomicAdd(cnt + (k >> fs), 1u)] = (uint16_t)(k & ((1u << PS) - 1));
        }
      }
    }
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(static_cast<uint16_t*>(P.item) + i0);
    const uint4* in = reinterpret_cast<const uint4*>(buf);
#pragma unroll
    for (uint32_t i = 0; i < PCHUNK * 2 / 16 / PT; ++i) out[i * PT + threadIdx.x] = in[i * PT + threadIdx.x];
    write_starts(P, stage, c, c0, c1);
  }
  __syncthreads();
  add_totals<true>(P, tot);
}

// Units of every range (one CTA per range; every CTA scans all ranges' unit
// counts).  A range of several units starts from zeroed bins (unless the
// counts add to those of an earlier round).
// (A range is 2^PS words of the result, words in all.)
//
// Units are cut by chunks, and pieces into parts of at least 64 items on
// average, as long as the range's keys are spread over its chunks.  Where they
// lie in lumps (a piece several times the average: sorted or sequential keys fill
// whole chunks with one range) its units are cut at equal numbers of keys
// instead, to the chunk, and their CTAs share every piece out over all warps;
// a range without keys is only stored.  (With the cuts by chunks alone one warp
// of a CTA, or one CTA of a range's, counted nearly all of such an input, and
// split pieces were walked where there were none.  256M keys over 16M bins,
// sorted 5.6 ms, in sequence 3.0, all the same 3.0: now 0.73 (0.62 with
// hk_look_kernel's choice), 0.77 and 0.62; 30M windows of N, 7 hashes into 1e6
// bits 1.36, now 0.24.)
template <typename W>
__global__ void __launch_bounds__(256) hk_plan_kernel(PartArgs P, uint64_t words, uint32_t unit_keys, uint32_t add,
                                                      W* __restrict__ out) {
  pdl_wait();
  if (P.cursor[2]) return;  // (no units: the cursors are cleared)
  __shared__ uint32_t s_before[8], s_all[8], s_mine;
  const uint32_t b = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t before = 0, all = 0, mine = 0;
  for (uint32_t r = threadIdx.x; r < P.ranges; r += 256) {
    const uint32_t u = max(1u, (P.total[r] + unit_keys - 1) / unit_keys);
    all += u;
    before += r < b ? u : 0;
    if (r == b) mine = u;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  all = __reduce_add_sync(0xffffffffu, all);
  if (lane == 0) s_before[warp] = before, s_all[warp] = all;
  if ((b & 255) == threadIdx.x) s_mine = mine;  // this thread met r == b
  __syncthreads();
  before = all = 0;
  for (int w = 0; w < 8; ++w) before += s_before[w], all += s_all[w];
  const uint32_t parts = s_mine, total = P.total[b], avg = total / P.chunks;
  uint32_t split = 0;
  while ((avg >> (split + 1)) >= 64) ++split;
  const bool lumps = (P.most[b] >> split) > max(4 * (avg >> split), 512u);
  uint32_t w = parts > 1 ? UNIT_SEVERAL : 0u;
  if (lumps) w |= UNIT_LUMPS;
  else w |= split << 8;
  if (lumps && parts > 1) {
    // unit i ends with the chunk in which the range's keys reach i + 1 parts of them
    const uint16_t* s0 = P.start + (uint64_t)b * P.chunks;
    const uint16_t* s1 = s0 + P.chunks;
    const uint32_t per = (P.chunks + 255) / 256, c0 = min(threadIdx.x * per, P.chunks), c1 = min(c0 + per, P.chunks);
    uint32_t sum = 0;
    for (uint32_t c = c0; c < c1; ++c) sum += s1[c] - s0[c];
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    __syncthreads();  // s_before has been read
    if (lane == 31) s_before[warp] = incl;
    __syncthreads();
    uint64_t at = incl - sum;
    for (int i = 0; i < warp; ++i) at += s_before[i];
    for (uint32_t i = threadIdx.x; i < parts; i += 256) P.unit[before + i].x = b, P.unit[before + i].w = w;
    if (threadIdx.x == 0) P.unit[before].y = 0, P.unit[before + parts - 1].z = P.chunks;
    for (uint32_t c = c0; c < c1; ++c) {
      const uint64_t end = at + (s1[c] - s0[c]);
      // the cuts i with at < i total / parts <= end
      for (uint64_t i = at * parts / total + 1; i < parts && i * total <= end * parts; ++i) {
        P.unit[before + i - 1].z = c + 1;
        P.unit[before + i].y = c + 1;
      }
      at = end;
    }
  } else {
    const uint32_t end = total ? P.chunks : 0u;
    const uint32_t per = ((end + parts - 1) / parts + 31) & ~31u;
    for (uint32_t i = threadIdx.x; i < parts; i += 256)
      P.unit[before + i] = make_uint4(b, min(i * per, end), min((i + 1) * per, end), w);
  }
  if (b == 0 && threadIdx.x == 0) {
    P.cursor[0] = 0;
    P.cursor[1] = all;
  }
  if (parts > 1 && !add)
    for (uint64_t i = ((uint64_t)b << PS) + threadIdx.x; i < ((uint64_t)(b + 1) << PS) && i < words; i += 256)
      out[i] = 0;
}

// A warp takes 32 parts at a time (a chunk's piece of the range is cut into
// 2^split parts, so that a unit of few chunks, of few ranges with long pieces,
// has work for every warp); they, in quads of four
// offsets (8 aligned bytes), are laid end to end and shared out evenly: quad f
// belongs to the part whose scanned quad count brackets it (a binary search
// over the lanes).  CAHEAD quads per lane are in flight (the pieces lie in
// DRAM).  A unit of lumps takes 1,024 pieces at a time, whose quads the whole CTA
// shares (the search is in shared memory).
constexpr int CAHEAD = 4;
// What is grouped, and what a range's words are: keys (16-bit bin numbers, u32
// counts, u64 results) or bit positions (32 bits, u32 words of a bit array).
struct KeyItems {
  using Item = uint16_t;
  using Quad = uint2;
  using Word = unsigned long long;
  static constexpr uint32_t CHUNK = PCHUNK;
  static constexpr bool LUMPS = true;
  static __device__ __forceinline__ void put(uint32_t* w, uint32_t x) { atomicAdd(w + x, 1u); }
  static __device__ __forceinline__ uint32_t item(const Quad& q, int i) {
    return (i & 1) ? (i < 2 ? q.x : q.y) >> 16 : (i < 2 ? q.x : q.y) & 0xffffu;
  }
  static __device__ __forceinline__ void add(Word* o, uint32_t v) { atomicAdd(o, (Word)v); }
  static __device__ __forceinline__ Word merged(Word o, uint32_t v) { return o + v; }
};
// Count CAHEAD quads per lane from quad f0 of `all` on: where(f, start, piece,
// chunk) gives the first quad, the piece (first offset | end << 16) and the
// chunk of the part that quad f belongs to; every lane calls it.
template <class T, class F>
__device__ __forceinline__ void count_quads(uint32_t* bins, const typename T::Item* items, uint32_t f0, uint32_t all,
                                            F&& where) {
  const uint32_t lane = threadIdx.x & 31;
  typename T::Quad w[CAHEAD];
  uint32_t r[CAHEAD], len[CAHEAD];  // the quad's first offset relative to its piece, and the piece's length
#pragma unroll
  for (int t = 0; t < CAHEAD; ++t) {
    const uint32_t f = f0 + 32 * t + lane;
    uint32_t first, pc, chunk;
    where(f, first, pc, chunk);
    const uint32_t i = 4 * (f - first) + (pc & 0xfffcu);
    r[t] = i - (pc & 0xffffu);
    len[t] = 0;
    if (f < all) {
      len[t] = (pc >> 16) - (pc & 0xffffu);
      w[t] = __ldg(reinterpret_cast<const typename T::Quad*>(items + (uint64_t)chunk * T::CHUNK + i));
    }
  }
#pragma unroll
  for (int t = 0; t < CAHEAD; ++t) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (r[t] + e < len[t]) T::put(bins, T::item(w[t], e));
  }
}

template <class T>
__global__ void __launch_bounds__(PCT, 1) hk_count_kernel(PartArgs P, uint64_t words, uint32_t add,
                                                          typename T::Word* __restrict__ out) {
  pdl_wait();
  const typename T::Item* items = static_cast<const typename T::Item*>(P.item);
  extern __shared__ __align__(16) uint32_t hc_bins[];  // [1 << PS]
  __shared__ uint32_t s_unit, s_ex[T::LUMPS ? PCT + 1 : 1], s_piece[T::LUMPS ? PCT : 1], wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nunits = P.cursor[1];
  for (;;) {
    __syncthreads();  // the previous unit's counts have been stored
    if (threadIdx.x == 0) s_unit = atomicAdd(P.cursor, 1u);
    for (uint32_t i = threadIdx.x; i < (1u << PS) / 4; i += PCT)
      reinterpret_cast<uint4*>(hc_bins)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if (s_unit >= nunits) return;
    const uint4 u = P.unit[s_unit];
    const uint16_t* s0 = P.start + (uint64_t)u.x * P.chunks;
    const uint16_t* s1 = s0 + P.chunks;
    if (T::LUMPS && (u.w & UNIT_LUMPS)) {
      for (uint32_t l0 = u.y; l0 < u.z; l0 += PCT) {
        const uint32_t c = l0 + threadIdx.x;
        uint32_t nq = 0;
        if (c < u.z) {
          const uint32_t a = s0[c], e = s1[c];
          if (e > a) nq = ((e + 3) >> 2) - (a >> 2), s_piece[threadIdx.x] = a | (e << 16);
        }
        s_ex[threadIdx.x] = nq;
        block_scan<PCT>(s_ex, PCT, wsum);
        const uint32_t all = s_ex[PCT];
        for (uint32_t f0 = 32 * CAHEAD * warp; f0 < all; f0 += PCT * CAHEAD)
          count_quads<T>(hc_bins, items, f0, all, [&](uint32_t f, uint32_t& first, uint32_t& pc, uint32_t& chunk) {
            uint32_t p = 0;  // the last piece that starts at quad f or before it
#pragma unroll
            for (uint32_t o = PCT / 2; o; o >>= 1)
              if (s_ex[p + o] <= f) p += o;
            first = s_ex[p], pc = f < all ? s_piece[p] : 0u, chunk = l0 + p;
          });
        __syncthreads();  // the pieces are counted
      }
    } else {
      const uint32_t split = u.w >> 8, nl = (u.z - u.y) << split;
      for (uint32_t l0 = 32 * warp; l0 < nl; l0 += PCT) {
        // this lane's piece: part `sub` of the quads of chunk c's
        const uint32_t l = l0 + lane, c = u.y + (l >> split), sub = l & ((1u << split) - 1);
        uint32_t piece = 0, nq = 0;  // first and end offset, quads
        if (l < nl) {
          const uint32_t a = s0[c], e = s1[c];
          const uint32_t qa = a >> 2, n4 = e > a ? ((e + 3) >> 2) - qa : 0;
          const uint32_t q0 = (n4 * sub) >> split, q1 = (n4 * (sub + 1)) >> split;
          nq = q1 - q0;
          if (nq) piece = max(a, 4 * (qa + q0)) | (min(e, 4 * (qa + q1)) << 16);
        }
        uint32_t ex = nq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t v = __shfl_up_sync(0xffffffffu, ex, o);
          if (lane >= o) ex += v;
        }
        const uint32_t all = __shfl_sync(0xffffffffu, ex, 31);
        ex -= nq;
        for (uint32_t f0 = 0; f0 < all; f0 += 32 * CAHEAD)
          count_quads<T>(hc_bins, items, f0, all, [&](uint32_t f, uint32_t& first, uint32_t& pc, uint32_t& chunk) {
            int p = 0;
#pragma unroll
            for (int o = 16; o; o >>= 1)
              if (__shfl_sync(0xffffffffu, ex, p + o) <= f) p += o;
            first = __shfl_sync(0xffffffffu, ex, p), pc = __shfl_sync(0xffffffffu, piece, p);
            chunk = u.y + ((l0 + p) >> split);
          });
      }
    }
    __syncthreads();
    const uint64_t b0 = (uint64_t)u.x << PS;
    const uint32_t nb = (uint32_t)min((uint64_t)(1u << PS), words - b0);
    for (uint32_t i = threadIdx.x; i < nb; i += PCT) {
      const uint32_t v = hc_bins[i];
      if (u.w & UNIT_SEVERAL) {
        if (v) T::add(out + b0 + i, v);
      } else {
        out[b0 + i] = add ? T::merged(out[b0 + i], v) : v;
      }
    }
  }
}

// ------------------------------------------------------------ Bloom filter
constexpr int BF_THREADS = 256;
constexpr int BF_TILE = 8192;                     // windows per CTA tile
constexpr int BF_WORDS = BF_TILE / 32 + 2;        // packed words: the tile plus up to 63 more bases

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// x mod m with r = floor((2^64 - 1) / m): q = floor(x r / 2^64) undershoots
// floor(x / m) by at most 2, so at most two corrections.
__device__ __forceinline__ uint64_t mod_barrett(uint64_t x, uint64_t m, uint64_t r) {
  const uint64_t q = __umul64hi(x, r);
  uint64_t rem = x - q * m;
  if (rem >= m) rem -= m;
  if (rem >= m) rem -= m;
  return rem;
}

// The same for m < 2^30: the remainder before the corrections is below 3 m, so
// its low 32 bits are all of it.
__device__ __forceinline__ uint32_t mod_barrett32(uint64_t x, uint32_t m, uint64_t r) {
  uint32_t rem = (uint32_t)x - (uint32_t)__umul64hi(x, r) * m;
  rem = min(rem, rem - m);  // (rem - m wraps to a large number when rem < m)
  return min(rem, rem - m);
}

// 2-bit code and invalid flag of 4 bases packed little-endian in w (first
// base in the low byte): codes A,C,G,T = 0..3 from bits 1..3 of the byte
// ((c >> 1) ^ (c >> 2)) & 3; big-endian 8-bit result (first base on top).
__device__ __forceinline__ void pack4(uint32_t w, uint32_t& code8, uint32_t& bad4) {
  const uint32_t ok = __vcmpeq4(w, 0x41414141u) | __vcmpeq4(w, 0x43434343u) | __vcmpeq4(w, 0x47474747u) |
                      __vcmpeq4(w, 0x54545454u);
  const uint32_t t = ((w >> 1) ^ (w >> 2)) & 0x03030303u;
  code8 = ((t & 3u) << 6) | (((t >> 8) & 3u) << 4) | (((t >> 16) & 3u) << 2) | ((t >> 24) & 3u);
  const uint32_t bad = ~ok;
  bad4 = ((bad & 1u) << 3) | (((bad >> 8) & 1u) << 2) | (((bad >> 16) & 1u) << 1) | ((bad >> 24) & 1u);
}

__global__ void __launch_bounds__(BF_THREADS)
bloom_kernel(const uint8_t* __restrict__ seq, uint64_t n, uint32_t L, uint64_t m, uint64_t rm, uint64_t rm1,
             uint32_t h, uint32_t* __restrict__ bits) {
  __shared__ unsigned long long sc[BF_WORDS];  // 32 bases per word, first base in the top bits
  __shared__ uint32_t sb[BF_WORDS];            // 1 = not A/C/G/T, same order
  if (n < L) return;
  const uint64_t nwin = n - L + 1;
  const uint64_t tiles = (nwin + BF_TILE - 1) / BF_TILE;
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t p0 = t * BF_TILE;
    __syncthreads();  // the previous tile's words are no longer read
    // pack bases p0 .. p0 + 32*BF_WORDS - 1 (beyond n: invalid)
    for (int wi = threadIdx.x; wi < BF_WORDS; wi += BF_THREADS) {
      uint64_t code = 0;
      uint32_t bad = 0;
      const uint64_t b0 = p0 + (uint64_t)wi * 32;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint64_t pos = b0 + (uint64_t)q * 4;
        uint32_t w = 0;
        if (pos + 4 <= n) {
          w = (uint32_t)seq[pos] | ((uint32_t)seq[pos + 1] << 8) | ((uint32_t)seq[pos + 2] << 16) |
              ((uint32_t)seq[pos + 3] << 24);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) w |= (pos + j < n ? (uint32_t)seq[pos + j] : 0u) << (8 * j);
        }
        uint32_t c8, b4;
        pack4(w, c8, b4);
        code = (code << 8) | c8;
        bad = (bad << 4) | b4;
      }
      sc[wi] = code;
      sb[wi] = bad;
    }
    __syncthreads();
    const uint64_t cnt = nwin - p0 < (uint64_t)BF_TILE ? nwin - p0 : (uint64_t)BF_TILE;
    for (uint32_t i = threadIdx.x; i < cnt; i += BF_THREADS) {
      const uint32_t wi = i >> 5, o = i & 31;
      const uint64_t bm = (((uint64_t)sb[wi] << 32) | sb[wi + 1]) << o;
      if (bm >> (64 - L)) continue;  // a base of the window is not A/C/G/T
      const uint64_t hi = sc[wi], lo = sc[wi + 1];
      const uint64_t cat = o ? (hi << (2 * o)) | (lo >> (64 - 2 * o)) : hi;
      const uint64_t code = cat >> (64 - 2 * L);
      uint64_t pos = mod_barrett(mix64(code), m, rm);
      const uint64_t step = 1 + mod_barrett(mix64(code ^ 0x9E3779B97F4A7C15ull), m - 1, rm1);
      for (uint32_t q = 0; q < h; ++q) {
        atomicOr(bits + (pos >> 5), 1u << (pos & 31));
        pos += step;
        if (pos >= m) pos -= m;
      }
    }
  }
}

// ----------------------------------------------------- partitioned filter
// The filter's atomicOrs are bound by the L2's atomic rate (210G bit-sets a
// second: 1.00 ms for 30M windows, 7 hashes), so, as for the large-key
// histogram, the positions of a job with many of them are grouped by ranges
// of 2^20 bits and each range is set in one CTA's shared memory and stored
// once.  A chunk is as many windows as have at most BCHUNK positions: they are
// computed once into shared memory (counting them by bucket), then grouped.
// 4 bytes a position are written and read again; 30M windows into 3e8 bits take
// 0.79 ms instead of 1.04 in all (grouping bound by issue and the shared-memory
// pipe), into 1e6 bits 0.82 instead of 2.16.
constexpr int BT = 1024;                 // threads of the grouping kernel (two CTAs per SM)
constexpr uint32_t BCHUNK = 16384;       // positions
constexpr uint32_t BNF = 512;            // buckets, at most
constexpr uint32_t BRANGES = 512;        // ranges, at most
constexpr uint32_t BS = PS + 5;          // log2 of a range's bits
constexpr uint32_t BNONE = 0xFFFFFFFFu;  // no position (m <= 2^29)
// Windows per chunk: as many whole warps of them as the chunk has room for, so
// that its positions take little more than the 4 bytes each that the interface
// states.  (Whole rounds of the CTA's threads filled chunks of 9 hashes to 56%,
// 7.2 bytes a position, and were slower: 30M windows into 3e8 bits, us a call,
// 5 hashes 624 / 608, 6 742 / 695, 7 829 / 788, 9 1,164 / 969, 12 1,302 / 1,243;
// into 1e6 bits 6 hashes 732 / 761, 9 1,161 / 1,061.)
__host__ __device__ constexpr uint32_t bloom_windows(uint32_t h) { return BCHUNK / h / 32 * 32; }
static_assert(bloom_windows(32) >= 32, "a chunk holds windows for every number of hashes");
struct BitItems {
  using Item = uint32_t;
  using Quad = uint4;
  using Word = uint32_t;
  static constexpr uint32_t CHUNK = BCHUNK;
  static constexpr bool LUMPS = false;  // (hashed)
  static __device__ __forceinline__ void put(uint32_t* w, uint32_t x) { atomicOr(w + (x >> 5), 1u << (x & 31)); }
  static __device__ __forceinline__ uint32_t item(const Quad& q, int i) { return key_at(q, i); }
  static __device__ __forceinline__ void add(Word* o, uint32_t v) { atomicOr(o, v); }
  static __device__ __forceinline__ Word merged(Word o, uint32_t v) { return o | v; }
};

// Four bases at pos (little-endian, beyond n: 0): two aligned words where both
// hold bases of the input, single bytes at its ends.
__device__ __forceinline__ uint32_t bases4(const uint8_t* __restrict__ seq, uint64_t n, uint64_t pos) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(seq + pos);
  const uint32_t sh = (uint32_t)(a & 3) * 8;
  if (pos + 8 <= n && pos >= 4) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(a & ~uintptr_t(3));
    return __funnelshift_r(__ldg(w), __ldg(w + 1), sh);
  }
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) v |= (pos + j < n ? (uint32_t)seq[pos + j] : 0u) << (8 * j);
  return v;
}

// Windows w0 .. w0 + nwin - 1 of the sequence, wt per chunk.
__global__ void __launch_bounds__(BT, 2) bloom_part_kernel(const uint8_t* __restrict__ seq, uint64_t n, uint64_t w0,
                                                           uint64_t nwin, uint32_t wt, uint32_t L, uint32_t m,
                                                           uint64_t rm, uint64_t rm1, uint32_t h, PartArgs P) {
  extern __shared__ __align__(16) unsigned char bp_sm[];
  uint32_t* pos = reinterpret_cast<uint32_t*>(bp_sm);             // [BCHUNK] in the order of the windows, then grouped
  uint32_t* cnt = pos + BCHUNK;                                   // [BNF + 1]
  uint32_t* tot = cnt + BNF + 4;                                  // [BRANGES]
  uint16_t* stage = reinterpret_cast<uint16_t*>(tot + BRANGES);   // [ranges + 1][PGROUP]
  __shared__ unsigned long long sc[BCHUNK / 32 + 2];  // 32 bases per word, first base in the top bits
  __shared__ uint32_t sb[BCHUNK / 32 + 2];            // 1 = not A/C/G/T, same order
  __shared__ uint32_t wsum[32];
  const uint32_t fs = P.fshift;
  for (uint32_t i = threadIdx.x; i < P.ranges; i += BT) tot[i] = 0;
  const uint32_t per = (P.chunks + gridDim.x - 1) / gridDim.x;
  const uint32_t c0 = blockIdx.x * per, c1 = min(c0 + per, P.chunks);
  for (uint32_t c = c0; c < c1; ++c) {
    const uint64_t first = (uint64_t)c * wt;
    const uint32_t count = first < nwin ? (uint32_t)min((uint64_t)wt, nwin - first) : 0;
    const uint64_t p0 = w0 + first;
    for (uint32_t i = threadIdx.x; i < P.nf; i += BT) cnt[i] = 0;
    // pack 8 bases per thread
    const uint32_t nw = count ? (count + L - 1 + 31) / 32 + 1 : 0;  // words, one of them past the last base
    for (uint32_t t = threadIdx.x; t < 4 * nw; t += BT) {
      uint32_t ca, ba, cb, bb;
      pack4(bases4(seq, n, p0 + 8 * t), ca, ba);
      pack4(bases4(seq, n, p0 + 8 * t + 4), cb, bb);
      const uint32_t wi = t >> 2, q = t & 3;
      reinterpret_cast<uint16_t*>(sc + wi)[3 - q] = (uint16_t)((ca << 8) | cb);
      reinterpret_cast<uint8_t*>(sb + wi)[3 - q] = (uint8_t)((ba << 4) | bb);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < count; i += BT) {
      const uint32_t wi = i >> 5, o = i & 31;
      const uint64_t bm = (((uint64_t)sb[wi] << 32) | sb[wi + 1]) << o;
      if (bm >> (64 - L)) {  // a base of the window is not A/C/G/T
        for (uint32_t q = 0; q < h; ++q) pos[q * count + i] = BNONE;
        continue;
      }
      const uint64_t hi = sc[wi], lo = sc[wi + 1];
      const uint64_t cat = o ? (hi << (2 * o)) | (lo >> (64 - 2 * o)) : hi;
      const uint64_t code = cat >> (64 - 2 * L);
      uint32_t x = mod_barrett32(mix64(code), m, rm);
      const uint32_t step = 1 + mod_barrett32(mix64(code ^ 0x9E3779B97F4A7C15ull), m - 1, rm1);
      uint32_t* at = pos + i;
#pragma unroll 4
      for (uint32_t q = 0; q < h; ++q, at += count) {
        *at = x;
        atomicAdd(cnt + (x >> fs), 1u);
        x += step;  // below 2^30
        x = min(x, x - m);
      }
    }
    __syncthreads();
    block_scan<BT>(cnt, P.nf, wsum);
    stage_starts<false>(P, cnt, stage, tot, c);
    const uint32_t all = cnt[P.nf], np = count * h;
    // grouped in place, from registers
    uint32_t x[BCHUNK / BT];
#pragma unroll
    for (int q = 0; q < (int)(BCHUNK / BT); ++q) {
      const uint32_t i = q * BT + threadIdx.x;
      x[q] = i < np ? pos[i] : BNONE;
    }
    __syncthreads();  // the starts and positions are read; the counters become cursors
#pragma unroll
    for (int q = 0; q < (int)(BCHUNK / BT); ++q)
      if (x[q] != BNONE) pos[atomicAdd(cnt + (x[q] >> fs), 1u)] = x[q] & ((1u << BS) - 1);
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(static_cast<uint32_t*>(P.item) + (uint64_t)c * BCHUNK);
    for (uint32_t i = threadIdx.x; i < (all + 3) / 4; i += BT) out[i] = reinterpret_cast<const uint4*>(pos)[i];
    __syncthreads();  // (the next chunk's positions go where these were)
    write_starts(P, stage, c, c0, c1);
  }
  __syncthreads();
  add_totals<false>(P, tot);
}

}  // namespace

int hk_smem_max_bins(const DevInfo& di) { return di.smem_optin / 4 - 1; }
int hk_cluster_max_bins(const DevInfo& di) { return HKC * (di.smem_optin / 4) - 1; }

template <typename C>
static cudaError_t launch_hk_cluster(const uint4* base, uint32_t off, uint64_t n, uint32_t nbins, C* cnt,
                                     const DevInfo& di, cudaStream_t s) {
  const uint32_t slice = (uint32_t)(((uint64_t)nbins + 1 + HKC - 1) / HKC);
  // multiply-high by floor(2^32 / slice) (at most 2^32 - 1) gives
  // floor(k / slice) or one less, for every k < 2^32
  const uint64_t sm64 = (1ull << 32) / slice;
  const uint32_t slice_mul = sm64 > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)sm64;
  const int bytes = (int)(slice * 4);
  cudaError_t e = allow_smem<hk_cluster_kernel<C>>(di);
  if (e != cudaSuccess) return e;
  const uint64_t groups = (n + off + 3) / 4;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = HKC;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(HK_SMEM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = (size_t)bytes;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // as many clusters as fit the GPU at once (each CTA holds one slice)
  int clusters = 0;
  cfg.gridDim = dim3(HKC, 1, 1);
  if ((e = cudaOccupancyMaxActiveClusters(&clusters, hk_cluster_kernel<C>, &cfg)) != cudaSuccess) return e;
  if (clusters < 1) return cudaErrorInvalidConfiguration;
  uint64_t want = (groups + (uint64_t)HK_SMEM_THREADS * 16 * HKC - 1) / ((uint64_t)HK_SMEM_THREADS * 16 * HKC);
  if (want < 1) want = 1;
  if (want > (uint64_t)clusters) want = (uint64_t)clusters;
  cfg.gridDim = dim3((unsigned)(want * HKC), 1, 1);
  return cudaLaunchKernelEx(&cfg, hk_cluster_kernel<C>, base, off, n, nbins, slice, slice_mul, cnt);
}

// Partitioned counting: chosen for MR_C_AUTO jobs whose bins do not fit one
// CTA, up to 2^25 bins (1,024 ranges), with at least a key per bin, from 2^24
// keys on, and from 2^22 when there are enough ranges for the counting kernel's
// CTAs (keys x ranges >= 2^26).  Measured, uniform / skewed keys, partitioned
// against the global array, us a call: 2^24 keys over 60,000 bins 143 / 146
// against 151 / 391; 2^23 over 60,000 124 / 124 against 91 / 211 (left to the
// array); 2^22 over 2^20 59 / 77 against 67 / 121; 2^24 over 2^24 123 / 366
// against 196 / 454; 2^28 over 30M 921 / 937 against 3,047 / 12,646.
constexpr uint64_t PART_ROUND = 1ull << 28;  // keys grouped at a time (2 bytes each of scratch)
bool hk_partitioned(uint64_t n, uint32_t nbins) {
  const uint64_t ranges = ((uint64_t)nbins >> PS) + 1;
  return ranges <= PRANGES && n >= nbins && (n >= 1ull << 24 || (n >= 1ull << 22 && n * ranges >= 1ull << 26));
}
// Scratch for `chunks` chunks, the result's words in ranges.
static PartArgs part_args(uint64_t chunks, uint32_t chunk_items, size_t item_bytes, uint32_t ranges, uint8_t* p,
                          size_t* bytes) {
  PartArgs P{};
  P.chunks = (uint32_t)((chunks + PGROUP - 1) / PGROUP * PGROUP);
  P.ranges = ranges;
  size_t at = 0;
  auto take = [&](size_t sz) {
    uint8_t* r = p + at;
    at += (sz + 255) & ~(size_t)255;
    return r;
  };
  P.item = take((size_t)P.chunks * chunk_items * item_bytes);
  P.start = reinterpret_cast<uint16_t*>(take((size_t)(P.ranges + 1) * P.chunks * 2));
  P.total = reinterpret_cast<uint32_t*>(take((size_t)(2 * P.ranges + 3) * 4));
  P.most = P.total + P.ranges;
  P.cursor = P.most + P.ranges;
  P.unit = reinterpret_cast<uint4*>(take((size_t)(2 * P.ranges + PUNITS) * 16));
  *bytes = at;
  return P;
}
static PartArgs hk_part_args(uint64_t n, uint32_t nbins, uint8_t* p, size_t* bytes) {
  const uint64_t m = n < PART_ROUND ? n : PART_ROUND;
  // + 3: keys may start inside a 16-byte group
  PartArgs P = part_args((m + 3 + PCHUNK - 1) / PCHUNK, PCHUNK, 2, (nbins >> PS) + 1, p, bytes);
  while (((nbins >> P.fshift) + 1) > PNF) ++P.fshift;
  P.nf = (nbins >> P.fshift) + 1;
  P.step = PS - P.fshift;
  return P;
}
size_t hk_part_bytes(uint64_t n, uint32_t nbins) {
  size_t b = 0;
  hk_part_args(n, nbins, nullptr, &b);
  return b;
}
cudaError_t launch_hist_keys_part(const uint32_t* keys, uint64_t n, uint32_t nbins, uint8_t* scratch,
                                  unsigned long long* out, const DevInfo& di, cudaStream_t s, uint64_t* nk,
                                  KTimer* kt) {
  size_t bytes = 0;
  const PartArgs P = hk_part_args(n, nbins, scratch, &bytes);
  const int psm = (int)(PCHUNK * 2 + (PNF + 4 + 2 * PRANGES) * 4 + (P.ranges + 1) * PGROUP * 2);
  const int csm = (1 << PS) * 4;
  cudaError_t e;
  if ((e = allow_smem<hk_part_kernel>(di)) != cudaSuccess ||
      (e = allow_smem<hk_count_kernel<KeyItems>>(di)) != cudaSuccess)
    return e;
  if ((e = kt_begin(kt, s)) != cudaSuccess) return e;
  for (uint64_t k0 = 0; k0 < n; k0 += PART_ROUND) {
    const uint64_t m = n - k0 < PART_ROUND ? n - k0 : PART_ROUND;
    const uintptr_t addr = reinterpret_cast<uintptr_t>(keys + k0);
    const uint4* base = reinterpret_cast<const uint4*>(addr & ~uintptr_t(15));
    const uint32_t off = (uint32_t)((addr & 15) / 4);
    const uint32_t pg = (uint32_t)di.sms * 2;
    const uint64_t uk = m / PUNITS > PUNIT_MIN ? m / PUNITS : PUNIT_MIN;
    const uint32_t add = k0 ? 1u : 0u;
    hk_look_kernel<<<di.sms, LOOK_T, 0, s>>>(base, m, P, (uint64_t)nbins + 1, add, out);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = launch_pdl(hk_part_kernel, dim3(P.chunks < pg ? P.chunks : pg), dim3(PT), (size_t)psm, s, base, off, m, nbins, P,
                        out)) != cudaSuccess ||
        (e = launch_pdl(hk_plan_kernel<unsigned long long>, dim3(P.ranges), dim3(256), 0, s, P, (uint64_t)nbins + 1,
                        (uint32_t)uk, add, out)) !=
            cudaSuccess ||
        (e = launch_pdl(hk_count_kernel<KeyItems>, dim3(di.sms), dim3(PCT), (size_t)csm, s, P, (uint64_t)nbins + 1, add,
                        out)) != cudaSuccess)
      return e;
    *nk += 4;
  }
  return kt_end(kt, s);
}

cudaError_t launch_hist_keys(const uint32_t* keys, uint64_t n, uint32_t nbins, int container, void* counters,
                             unsigned long long* out, const DevInfo& di, cudaStream_t s, uint64_t* nk, KTimer* kt) {
  const bool smem = container == MR_C_SMEM_ARRAY, wide = smem || !counters;
  const uint64_t nb = (uint64_t)nbins + 1;
  cudaError_t e = cudaMemsetAsync(wide ? (void*)out : counters, 0, nb * (wide ? 8 : 4), s);
  if (e != cudaSuccess) return e;
  const uintptr_t addr = reinterpret_cast<uintptr_t>(keys);
  const uint4* base = reinterpret_cast<const uint4*>(addr & ~uintptr_t(15));
  const uint32_t off = (uint32_t)((addr & 15) / 4);
  const uint64_t groups = (n + off + 3) / 4;
  if (n) {
    if ((e = kt_begin(kt, s)) != cudaSuccess) return e;
    if (smem) {
      const int bytes = (int)(nb * 4);
      const int per_sm = bytes <= 48 * 1024 ? 2 : 1;
      uint64_t g = (groups + HK_SMEM_THREADS * 16 - 1) / (HK_SMEM_THREADS * 16);
      g = g < 1 ? 1 : g;
      g = g > (uint64_t)di.sms * per_sm ? (uint64_t)di.sms * per_sm : g;
      if ((e = allow_smem<hk_smem_kernel>(di)) != cudaSuccess) return e;
      hk_smem_kernel<<<(int)g, HK_SMEM_THREADS, bytes, s>>>(base, off, n, nbins, out);
    } else if (container == MR_C_CLUSTER_ARRAY) {
      e = wide ? launch_hk_cluster(base, off, n, nbins, out, di, s)
               : launch_hk_cluster(base, off, n, nbins, static_cast<uint32_t*>(counters), di, s);
      if (e != cudaSuccess) return e;
    } else {
      uint64_t g = (groups + HK_THREADS * 8 - 1) / (HK_THREADS * 8);
      g = g < 1 ? 1 : g;
      g = g > (uint64_t)di.sms * 8 ? (uint64_t)di.sms * 8 : g;
      if (wide)
        hk_global_kernel<unsigned long long><<<(int)g, HK_THREADS, 0, s>>>(base, off, n, nbins, out);
      else
        hk_global_kernel<uint32_t><<<(int)g, HK_THREADS, 0, s>>>(base, off, n, nbins, static_cast<uint32_t*>(counters));
    }
    if ((e = cudaGetLastError()) != cudaSuccess || (e = kt_end(kt, s)) != cudaSuccess) return e;
    ++*nk;
  }
  if (!wide) {
    uint64_t g = (nb + 1023) / 1024;
    g = g > (uint64_t)di.sms * 8 ? (uint64_t)di.sms * 8 : (g < 1 ? 1 : g);
    hk_widen_kernel<<<(int)g, 1024, 0, s>>>(static_cast<const uint32_t*>(counters), nb, out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ++*nk;
  }
  return cudaSuccess;
}

cudaError_t launch_bloom(const uint8_t* seq, uint64_t n, uint32_t L, uint64_t m, uint32_t h, uint32_t* bits,
                         const DevInfo& di, cudaStream_t s, uint64_t* nk, KTimer* kt) {
  const uint64_t words = (m + 31) / 32;
  cudaError_t e = cudaMemsetAsync(bits, 0, words * 4, s);
  if (e != cudaSuccess || n < L) return e;
  const uint64_t rm = ~0ull / m, rm1 = ~0ull / (m - 1);
  const uint64_t tiles = (n - L + 1 + BF_TILE - 1) / BF_TILE;
  uint64_t g = tiles < (uint64_t)di.sms * 8 ? tiles : (uint64_t)di.sms * 8;
  if ((e = kt_begin(kt, s)) != cudaSuccess) return e;
  bloom_kernel<<<(int)g, BF_THREADS, 0, s>>>(seq, n, L, m, rm, rm1, h, bits);
  if ((e = cudaGetLastError()) != cudaSuccess || (e = kt_end(kt, s)) != cudaSuccess) return e;
  ++*nk;
  return cudaSuccess;
}

// Partitioned filter: up to 2^29 bits (512 ranges), from 2^24 positions on, with
// at least 5 hashes (the two 64-bit mixes of a window are paid once) or few
// ranges, whose words the L2's atomics contend for.  Measured, partitioned
// against atomicOr on the global array, us a call: 30M windows x 7 into 3e8
// bits 788 / 1,040, x 3 into 2.4e8 500 / 465 (left to the array), x 3 into 1e6 472 / 944;
// 3M x 7 into 2.4e7 124 / 144; 5.6M x 3 into 1e6 155 / 203.
constexpr uint64_t BLOOM_ROUND = 1ull << 29;  // positions grouped at a time (4 bytes each of scratch, and gaps of at most 6%)
bool bloom_partitioned(uint64_t n, uint32_t L, uint64_t m, uint32_t h) {
  return n >= L && m <= (uint64_t)BRANGES << BS && (n - L + 1) * h >= 1ull << 24 && (h >= 5 || m <= 1ull << 24);
}
static uint64_t bloom_round(uint32_t h) { return BLOOM_ROUND / BCHUNK * bloom_windows(h); }  // windows grouped at a time
static PartArgs bloom_part_args(uint64_t n, uint32_t L, uint64_t m, uint32_t h, uint8_t* p, size_t* bytes) {
  const uint64_t nwin = n - L + 1, w = nwin < bloom_round(h) ? nwin : bloom_round(h);
  const uint32_t wt = bloom_windows(h);
  PartArgs P = part_args((w + wt - 1) / wt, BCHUNK, 4, (uint32_t)((m - 1) >> BS) + 1, p, bytes);
  while (((m - 1) >> P.fshift) + 1 > BNF) ++P.fshift;
  P.nf = (uint32_t)((m - 1) >> P.fshift) + 1;
  P.step = BS - P.fshift;
  return P;
}
size_t bloom_part_bytes(uint64_t n, uint32_t L, uint64_t m, uint32_t h) {
  size_t b = 0;
  bloom_part_args(n, L, m, h, nullptr, &b);
  return b;
}
cudaError_t launch_bloom_part(const uint8_t* seq, uint64_t n, uint32_t L, uint64_t m, uint32_t h, uint8_t* scratch,
                              uint32_t* bits, const DevInfo& di, cudaStream_t s, uint64_t* nk, KTimer* kt) {
  size_t bytes = 0;
  const PartArgs P = bloom_part_args(n, L, m, h, scratch, &bytes);
  const int psm = (int)((BCHUNK + BNF + 4 + BRANGES) * 4 + (P.ranges + 1) * PGROUP * 2);
  const int csm = (1 << PS) * 4;
  const uint64_t words = (m + 31) / 32, nwin = n - L + 1, rm = ~0ull / m, rm1 = ~0ull / (m - 1);
  cudaError_t e;
  if ((e = allow_smem<bloom_part_kernel>(di)) != cudaSuccess ||
      (e = allow_smem<hk_count_kernel<BitItems>>(di)) != cudaSuccess)
    return e;
  if ((e = kt_begin(kt, s)) != cudaSuccess) return e;
  for (uint64_t w0 = 0; w0 < nwin; w0 += bloom_round(h)) {
    const uint64_t w = nwin - w0 < bloom_round(h) ? nwin - w0 : bloom_round(h);
    const uint64_t uk = w * h / PUNITS > PUNIT_MIN ? w * h / PUNITS : PUNIT_MIN;
    const uint32_t add = w0 ? 1u : 0u, pg = (uint32_t)di.sms * 2;
    if ((e = cudaMemsetAsync(P.total, 0, (2 * P.ranges + 3) * 4, s)) != cudaSuccess) return e;
    bloom_part_kernel<<<P.chunks < pg ? P.chunks : pg, BT, psm, s>>>(seq, n, w0, w, bloom_windows(h), L, (uint32_t)m, rm,
                                                                     rm1, h, P);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = launch_pdl(hk_plan_kernel<uint32_t>, dim3(P.ranges), dim3(256), 0, s, P, words, (uint32_t)uk, add,
                        bits)) != cudaSuccess ||
        (e = launch_pdl(hk_count_kernel<BitItems>, dim3(di.sms), dim3(PCT), (size_t)csm, s, P, words, add, bits)) !=
            cudaSuccess)
      return e;
    *nk += 3;
  }
  return kt_end(kt, s);
}

}  // namespace mrgb
