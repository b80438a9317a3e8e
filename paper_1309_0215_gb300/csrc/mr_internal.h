// Internal declarations shared by the CUDA translation units of libmrgb.so.
#pragma once
#include <atomic>
#include <utility>
#include <cuda_runtime.h>
#include <cstdint>
#include <cstddef>

#include "../../include/mr.h"
#include "dev_wordcount.cuh"

namespace mrgb {

// ---------------------------------------------------------------- helpers
void set_last_error(const char* where, cudaError_t e);

#define MR_CUDA_TRY(expr)                                   \
  do {                                                      \
    cudaError_t e_ = (expr);                                \
    if (e_ != cudaSuccess) {                                \
      ::mrgb::set_last_error(#expr, e_);                    \
      return MR_ECUDA;                                      \
    }                                                       \
  } while (0)

struct DevInfo {
  int sms = 0;
  int smem_optin = 0;   // max dynamic shared memory per block (opt-in)
  int l2_bytes = 0;
};

#ifdef __CUDACC__
// Lets KERN be launched with any dynamic shared memory a CTA of the device can
// have.  The limit is an attribute of the function on the device, shared by all
// contexts and threads, and nothing holds it between a launcher's setting it and
// its launches: every launcher sets the same value, never its own job's size,
// which another thread's larger job would then exceed.
template <auto KERN>
inline cudaError_t allow_smem(const DevInfo& di) {
  static std::atomic<int> fixed{-1};  // the kernel's static shared memory
  int f = fixed.load(std::memory_order_relaxed);
  if (f < 0) {
    cudaFuncAttributes a{};
    const cudaError_t e = cudaFuncGetAttributes(&a, KERN);
    if (e != cudaSuccess) return e;
    fixed.store(f = (int)a.sharedSizeBytes, std::memory_order_relaxed);
  }
  return cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, di.smem_optin - f);
}
#endif

// ------------------------------------------------------------ array jobs
// RGB8 histogram, local arrays in shared memory ("lane-column" layout:
// bins x 32 u32 columns, one column per lane, shared by all warps of a CTA).
// bins must be zeroed before the launch.
cudaError_t launch_hist_smem(const uint8_t* in, uint64_t n, uint64_t* bins, int grid, cudaStream_t s);
// RGB8 histogram without local arrays: atomics straight on the global bins.
cudaError_t launch_hist_global(const uint8_t* in, uint64_t n, uint64_t* bins, int grid, cudaStream_t s);
// int8 regression sums; sums must be zeroed before the launch.
cudaError_t launch_linreg(const int8_t* in, uint64_t n, int64_t* sums, int grid, cudaStream_t s);
// Independent array jobs run as one launch (shared-memory histograms and
// regressions; at most ARRAY_FUSE_MAX).
constexpr int ARRAY_FUSE_MAX = 8;
struct ArrayJobs {
  uint32_t n;
  uint32_t kind[ARRAY_FUSE_MAX];
  const uint8_t* in[ARRAY_FUSE_MAX];
  uint64_t bytes[ARRAY_FUSE_MAX];
  void* out[ARRAY_FUSE_MAX];
};
cudaError_t launch_array_fused(const ArrayJobs& jobs, int grid, cudaStream_t s);

int hist_smem_bytes();         // dynamic shared memory the smem histogram needs
int hist_block_threads();

// ------------------------------------------------------ kernel timing
// Event pairs around each launch of a job's main kernel (the distance pass of
// every k-means iteration, the word-count map pass, the one counting kernel of
// the other kinds), recorded when the context times its jobs.  Events are
// created on first use; launches past MAX are not timed.
struct KTimer {
  static constexpr uint32_t MAX = 64;
  cudaEvent_t ev[2 * MAX] = {};
  uint32_t n = 0;  // launches timed in the current run
};
cudaError_t kt_begin(KTimer* t, cudaStream_t s);  // no-op for t == nullptr
cudaError_t kt_end(KTimer* t, cudaStream_t s);
void kt_destroy(KTimer* t);

// ------------------------------------------- large-key histogram, Bloom
// Largest bin count whose local arrays (nbins + 1 u32) fit one CTA, and a
// thread-block cluster of CTAs.
int hk_smem_max_bins(const DevInfo& di);
int hk_cluster_max_bins(const DevInfo& di);
// Histogram of n u32 keys into out[nbins + 1] (zeroed here).  container:
// MR_C_SMEM_ARRAY local arrays per CTA, MR_C_CLUSTER_ARRAY local arrays
// spread over a cluster's shared memory, else atomics on the global array.
// Local arrays of one CTA go straight into the u64 output; the other containers
// count in the u32 counters (nbins + 1 words) and widen at the end, or straight
// into the output without counters (null, as from 2^32 keys on).
cudaError_t launch_hist_keys(const uint32_t* keys, uint64_t n, uint32_t nbins, int container, void* counters,
                             unsigned long long* out, const DevInfo& di, cudaStream_t s, uint64_t* nk,
                             KTimer* kt = nullptr);
// The same for many keys over bins beyond one CTA's shared memory
// (hk_partitioned), through hk_part_bytes of scratch; every bin is written.
bool hk_partitioned(uint64_t n, uint32_t nbins);
size_t hk_part_bytes(uint64_t n, uint32_t nbins);
cudaError_t launch_hist_keys_part(const uint32_t* keys, uint64_t n, uint32_t nbins, uint8_t* scratch,
                                  unsigned long long* out, const DevInfo& di, cudaStream_t s, uint64_t* nk,
                                  KTimer* kt = nullptr);
// Bloom-filter build over n bases into ceil(m / 32) u32 words (zeroed here).
cudaError_t launch_bloom(const uint8_t* seq, uint64_t n, uint32_t L, uint64_t m, uint32_t h, uint32_t* bits,
                         const DevInfo& di, cudaStream_t s, uint64_t* nk, KTimer* kt = nullptr);

// The same for many positions (bloom_partitioned), through bloom_part_bytes of
// scratch; every word is written.
bool bloom_partitioned(uint64_t n, uint32_t L, uint64_t m, uint32_t h);
size_t bloom_part_bytes(uint64_t n, uint32_t L, uint64_t m, uint32_t h);
cudaError_t launch_bloom_part(const uint8_t* seq, uint64_t n, uint32_t L, uint64_t m, uint32_t h, uint8_t* scratch,
                              uint32_t* bits, const DevInfo& di, cudaStream_t s, uint64_t* nk, KTimer* kt = nullptr);

// --------------------------------------------------------- word count job
struct WcBuffers {
  uint64_t cap = 0;            // global hash-table slots (power of two)
  uint64_t* key = nullptr;     // [cap][2] 128-bit keys, {0, 0} = empty
  uint64_t* cnt = nullptr;     // [cap] combined counts (contiguous after key)
  uint32_t* state = nullptr;   // 64 bytes: word 0 overflow flag, 64-bit fields 1..4 post-phase bounds
  uint8_t* sortbuf = nullptr;  // post-phase scratch for cap records
  uint64_t* host = nullptr;    // pinned host words {flags, records, key bytes}, written by the last kernel (or null)
  bool one_cta = false;        // a small text may take the one-CTA kernel (automatic tables)
  uint8_t* out = nullptr;      // result: header + records + key bytes
  uint64_t out_cap = 0;
};
uint64_t wc_table_bytes(uint64_t cap);
uint64_t wc_state_bytes();
size_t wc_sortbuf_bytes(uint64_t records);
uint64_t wc_out_bytes(uint64_t cap, uint64_t n);
int wc_map_smem_bytes();
uint64_t wc_compact_blocks(uint64_t cap);
wc::JobDev wc_job_dev(const uint8_t* in, uint64_t n, const WcBuffers& b, uint64_t blk0);
// Compaction, sort (by job, count desc, key asc), bounds and gather for
// njobs jobs (jobs: device array, or nullptr for one job; hjobs: the same
// descriptors in host memory, njobs of them).  sms sizes persistent grids.
cudaError_t launch_wordcount_post_multi(const wc::JobDev* jobs, const wc::JobDev* hjobs, uint32_t njobs,
                                        uint64_t nblocks, uint64_t records, uint8_t* sortbuf, int sms,
                                        cudaStream_t s, uint64_t* nk);
// Zero the table and state, run map+combine, compaction, sort and gather.
// *nk is incremented by the number of kernels launched.
// pipelined: the map pass runs as mapper warps handing cache misses to
// reducer warps through shared-memory rings (wc_pipe_kernel).
// pipe_polls: polls of the pipelined pass's bounded ring waits (< 0: default).
cudaError_t launch_wordcount(const uint8_t* in, uint64_t n, const WcBuffers& b, const DevInfo& di, cudaStream_t s,
                             uint64_t* nk, bool pipelined = false, KTimer* kt = nullptr, long long pipe_polls = -1);

// ---------------------------------------------------------------- k-means
// Programmatic dependent launch: the kernel may be scheduled while the
// kernel before it on the stream is still finishing (its launch and ramp
// overlap that kernel's tail); it must call pdl_wait() before touching any
// memory, which returns once the earlier kernel has completed and its writes
// are visible.  Used only for kernels that start with pdl_wait() and follow
// another kernel on the stream.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}
// Distance bounds that let later rounds skip points (see km_filter_kernel).
struct KmBounds {
  float* ub = nullptr;           // [n] upper bound on the distance to the own centroid, less that centroid's drift so far
  float* lb = nullptr;           // [n] lower bound on the distance to any other, plus the largest drifts so far
  const float* drift = nullptr;  // [k] each centroid's drift so far
  const float* far = nullptr;    // [1] the sum of the rounds' largest drifts
  const uint32_t* mode = nullptr;  // [1] KM_FILTER, KM_BOUNDS or KM_REST: what the round does
};
// The filter at work; the pass over all points with the bounds written, for the
// filter of the next round; neither (see km_filter_kernel).
constexpr uint32_t KM_FILTER = 0, KM_BOUNDS = 1, KM_REST = 2;

// A point with 2 to KM_CAND_MAX candidate centroids, 12 bits each (K <= 4096),
// and their number in the top bits.
constexpr uint32_t KM_CAND_MAX = 5;
struct KmFew {
  uint32_t p, lo, hi;
};
#ifdef __CUDACC__
__device__ __forceinline__ KmFew km_few(uint32_t p, uint64_t cand, uint32_t ncand) {
  return KmFew{p, (uint32_t)cand, ((uint32_t)(cand >> 32) & 0x0FFFFFFFu) | (ncand << 28)};
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// An assignment word holds the point's cluster (low half) and the cluster it
// had when the sums were last updated (high half; K <= 4096).
__device__ __forceinline__ uint32_t km_word(uint32_t now, uint32_t summed) { return now | (summed << 16); }
// Both, for indexing: a word that a timed-out pass left unwritten counts as cluster 0.
__device__ __forceinline__ uint32_t km_now(uint32_t w, uint32_t k) { return (w & 0xffffu) < k ? w & 0xffffu : 0u; }
// Bounds of point p from squared distances: at most u2 to its centroid, whose
// drift so far is given, at least l2 to every other (sqrt.approx and the sums
// below are good to a few units in the last place, 1e-6 is eight).
__device__ __forceinline__ float km_sqrt(float v) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ void km_put_bounds(const KmBounds& B, uint32_t p, float drift, float far, float u2,
                                              float l2) {
  B.ub[p] = fmaf(km_sqrt(u2), 1.000001f, -drift);
  B.lb[p] = fmaf(km_sqrt(fmaxf(l2, 0.f)), 0.999999f, far);
}
__device__ __forceinline__ bool km_keeps_bounds(const KmBounds& B) { return B.ub && *B.mode != KM_REST; }
__device__ __forceinline__ uint32_t km_summed(uint32_t w, uint32_t k) { return (w >> 16) < k ? w >> 16 : 0u; }
#endif

struct KmBuffers {
  uint32_t n = 0, d = 0, k = 0;
  float* cent = nullptr;        // [k][d] current centroids (FP32 state)
  uint32_t* assign = nullptr;   // [n] assignment words (km_word)
  long long* sums = nullptr;    // [k][d] fixed-point sums
  unsigned long long* counts = nullptr;  // [k] cluster sizes, then [k] those a full update counts
  unsigned long long* stats = nullptr;   // [4]
  uint32_t* flagged = nullptr;  // [n] points to re-check; later the sorted update's permutation
  uint32_t* nflag = nullptr;    // [8] counters: [1] points to re-check, [2] max|x| bits, [4] pairs; of even and odd
                                //     rounds: [0], [5] points that changed cluster, [6], [7] max||c|| bits
  KmFew* pairs = nullptr;       // [n] points with a few candidate centroids
  float* cnorm = nullptr;       // [k] ||c||^2 (of the shifted centroids on the tensor-core path)
  float* center = nullptr;      // [d] the shift (nullptr where no tensor-core pass covers the shape)
  unsigned int* maxabs = nullptr;  // [1] bits of max |x|
  int* shift = nullptr;         // [1] fixed-point scale exponent
  KmBounds bounds;              // ub nullptr: not kept
  float* half = nullptr;        // [k] half the distance to the nearest other centroid
  uint32_t* act = nullptr;      // [n] points whose distances the round computes
  uint64_t* host = nullptr;     // pinned host word for the count of timed-out waits, written by the last kernel (or null)
  uint8_t* bop = nullptr;       // centroid operands of the wide tensor-core pass (nullptr: not taken)
  uint32_t* kcursor = nullptr;  // [k] counting-sort write cursors, in the norms' place
  long long* part = nullptr;    // [CTAs][k][d] partial sums of the local-array update (nullptr: sort path)
  KTimer* kt = nullptr;         // times the distance pass of each iteration
  int precision = 0;
  // diagnostics (mr_set_option): polls of a bounded device wait (< 0: the
  // default), cap on the CTAs of the persistent kernels (0: none), tiles the
  // tensor-core kernel's bulk-copy thread stages per CTA (0: all)
  long long polls = -1;
  uint32_t grid_cap = 0;
  uint32_t stop_copies = 0;
};
// wide: with the wide tensor-core pass's operands
size_t km_scratch_bytes(uint32_t n, uint32_t d, uint32_t k, bool wide);
cudaError_t km_carve(KmBuffers& b, uint8_t* base, size_t bytes, bool wide);
// the filter's bounds, in memory of their own (after km_carve)
bool km_bounds_pay(uint32_t n, uint32_t k, uint32_t iters);
size_t km_bounds_bytes(uint32_t n, uint32_t k);
void km_carve_bounds(KmBuffers& b, uint8_t* base);
cudaError_t launch_kmeans(const float* x, const float* init, uint32_t iters, KmBuffers& b, const DevInfo& di,
                          cudaStream_t s, float* out_cent, int32_t* out_assign, unsigned long long* out_stats,
                          uint64_t* nk);
bool km_tc_supported(uint32_t d, uint32_t k);
bool km_wide_supported(uint32_t d, uint32_t k);
size_t km_wide_operand_bytes(uint32_t d, uint32_t k);

// --------------------------------------------------------- batched launch
struct BatchJob {
  uint32_t kind;       // mr_kind
  uint32_t container;  // mr_container chosen
  const uint8_t* in;
  uint64_t n;
  void* out;           // histogram bins / regression sums
  wc::JobDev wc;       // word count
  uint64_t tile_begin; // first tile index of this job in the batch's tile space
  uint64_t ntiles;
  uint64_t zchunk0;    // first clearing chunk of this job's container (batch_zero_chunks)
};
cudaError_t batch_prepare();
// Zero the jobs' containers (total_zchunks chunks, see batch_zero_chunks),
// then run every tile in one persistent launch.
cudaError_t launch_batch(const BatchJob* jobs_dev, uint32_t njobs, uint64_t total_tiles, unsigned long long* cursor,
                         uint64_t arr_tile, uint64_t wc_tile, uint64_t total_zchunks, const DevInfo& di,
                         cudaStream_t s, uint64_t* nk);
uint64_t batch_tiles_for(uint32_t kind, uint64_t n, uint64_t arr_tile, uint64_t wc_tile);
// Chunks of BATCH_ZCHUNK bytes that clearing the job's container takes.
constexpr uint64_t BATCH_ZCHUNK = 64 * 1024;
uint64_t batch_zero_chunks(uint32_t kind, uint64_t wc_cap);

}  // namespace mrgb
