// Device code of the word-count map + combine pass, shared by the plain
// kernel (k_wordcount.cu) and the persistent batched kernel (k_batch.cu).
//
// Map (arXiv:1309.0215 Sec. II-A): a token is a maximal run of bytes that are
// not ASCII whitespace; each emits (token, 1); reduce is a sum.
//
// Key encoding (128 bits, the container's key):
//   short token, 1..15 bytes:  w0 = bytes 0..7 (little-endian, zero padded)
//                              w1 = bytes 8..14 | length << 56
//   long token, >= 16 bytes:   w0 = offset of an occurrence in the input + 1
//                              w1 = 0xFF << 56 | length
// A short key is its own identity (no memory read to compare); a long key
// is compared byte for byte against the resident, immutable input.  w1 is
// never zero, so {0, 0} marks an empty slot.
//
// Global container: open addressing, linear probing, a slot = 16-byte key
// claimed with one 128-bit atomic CAS (written once, never changed) plus a
// 64-bit count updated with atomicAdd.  Running out of probes raises the
// job's overflow flag (the host then re-runs with a larger table).
//
// Local container (the paper's combiner, Sec. III-A, with the bounded local
// table of Sec. III-D), shaped for Zipf-like key streams: a 2-way cache of
// hot keys per warp in shared memory (two candidate slots per key, one
// compare each, no probing) absorbs the frequent keys, and the rest go
// straight to the global container, where such rarer keys do not contend.
// No warp collective is used: lanes of one round that carry the same key
// simply add to the same slot count (shared-memory atomics), and an empty
// slot is claimed with a 64-bit shared-memory CAS.  The cache is merged into
// the global container every CACHE_EPOCH segments (so it can re-learn which
// keys are hot) and at the end.
#pragma once
#include <cstdint>

namespace mrgb {
namespace wc {

constexpr int SEG = 512;                // bytes per warp step (16 per lane), but for MapWarp
constexpr int HALO = 32;                // staged bytes after the segment (a token's first 16 and word loads)
constexpr int LT = 128;                 // hot-key cache entries per warp
constexpr int CACHE_EPOCH = 64;         // segments between cache merges
constexpr int MAX_PROBES = 4096;
constexpr uint64_t LONG_TAG = 0xFFull << 56;
constexpr uint64_t LEN_MASK = (1ull << 56) - 1;

struct WarpLocal {
  static constexpr int LANE = 16;  // bytes of the segment per lane
  unsigned long long w0[LT];
  unsigned long long w1[LT];
  uint32_t h[LT];
  uint32_t cnt[LT];
  uint8_t buf[SEG + HALO];
  uint16_t starts[SEG / 2];    // the tokens: first byte | length << 12 (0: 16 bytes or more)
};
static_assert(sizeof(WarpLocal) % 16 == 0, "WarpLocal must keep 16-byte alignment");

// One word-count job as the kernels see it.
struct JobDev {
  const uint8_t* in;
  uint64_t n;
  unsigned long long* key;   // [cap][2]
  unsigned long long* cnt;   // [cap]
  uint64_t cap;              // power of two
  uint32_t log2cap;
  uint32_t* state;           // [0] overflow flag; [2..7] filled by the post phase
  uint8_t* out;
  uint64_t blk0;             // first compaction block of this job
  uint64_t* host;            // host memory for {flags, records, key bytes}, written by the last kernel; or null
};

__device__ __forceinline__ bool is_ws(uint32_t c) { return c == 32u || (c - 9u) < 5u; }

// 0x80 in every byte of u that is ASCII whitespace (0x20, or 0x09..0x0D),
// else 0: exact per byte, with no carry between bytes.  Space: the byte of
// u ^ 0x20202020 is zero iff ((b & 0x7F) + 0x7F) | b has its top bit clear.
// 9..13: with h = b & 0x7F, h + 0x77 reaches 0x80 iff h >= 9 and h + 0x72
// iff h >= 14; bytes >= 0x80 are excluded by their own top bit.
__device__ __forceinline__ uint32_t ws_bytes(uint32_t u) {
  const uint32_t x = u ^ 0x20202020u;
  const uint32_t sp = ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x);
  const uint32_t h = u & 0x7F7F7F7Fu;
  const uint32_t rg = (h + 0x77777777u) & ~(h + 0x72727272u) & ~u;
  return (sp | rg) & 0x80808080u;
}
// compress ws_bytes' mask to 4 bits (byte i -> bit i)
__device__ __forceinline__ uint32_t byte_bits(uint32_t m) { return (m * 0x00204081u) >> 28; }
// The 16 whitespace bits of 16 bytes: four dot products of the byte masks with
// powers of two (each sum is 128 times eight bits).
__device__ __forceinline__ uint32_t ws_bits(const uint4& v) {
  const uint32_t lo = __dp4a(ws_bytes(v.y), 0x80402010u, __dp4a(ws_bytes(v.x), 0x08040201u, 0u));
  const uint32_t hi = __dp4a(ws_bytes(v.w), 0x80402010u, __dp4a(ws_bytes(v.z), 0x08040201u, 0u));
  return (lo >> 7) | (hi << 1);
}
// the low n bits of v (n <= 0: none; n >= 32: all)
__device__ __forceinline__ uint32_t low_bits(uint32_t v, int n) {
  uint32_t r;
  asm("szext.clamp.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"((uint32_t)(n > 0 ? n : 0)));
  return r;
}

__device__ __forceinline__ uint64_t fmix64(uint64_t k) {
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

// 32-bit mix of the four 32-bit words of a short key (the key is compared
// exactly; the hash only spreads slots): NH (Black, Halevi, Krawczyk, Krovetz and
// Rogaway, "UMAC", 1999), two 64-bit products of the words with constants added,
// folded to 32 bits.  The products have to be that wide: the low half of one
// drops what lies above it, so that keys which differ in the last byte of each
// word, such as 12-byte keys in three groups of four, would meet at 256 values.
// (Any three bytes of 15 varied over 40 values: at least 0.9995 of the keys have
// a hash of their own.  Four multiply-adds of 32 x 64 bits in place of the two
// products took 417 us for 256 MB of 50,000 words, this 410; the 32-bit sum 407.)
// The constants are primes of xxHash32 (Collet) with the third byte DF: a word
// whose sum with one is zero, and whose product would forget the other word, has
// 20 as its third byte, a space, or as the last word a length above 15.  The
// last multiplier is of MurmurHash3's finalizer (Appleby), whose 64-bit form
// fmix64 is.
__device__ __forceinline__ uint32_t hash_short(uint32_t u0, uint32_t u1, uint32_t u2, uint32_t u3) {
  const uint64_t t =
      (uint64_t)(u0 + 0x9EDF79B1u) * (u1 + 0x85DFCA77u) + (uint64_t)(u2 + 0xC2DFAE3Du) * (u3 + 0x27D4EB2Fu);
  uint32_t h = ((uint32_t)t ^ (uint32_t)(t >> 32)) * 0x85EBCA6Bu;
  h ^= h >> 15;
  return h;
}

struct Tok {
  uint64_t w0, w1;
  uint32_t h;
};

// Bytes of two long tokens of equal length len, at offsets a and b.
__device__ inline bool long_equal(const uint8_t* __restrict__ in, uint64_t a, uint64_t b, uint64_t len) {
  if (a == b) return true;
  for (uint64_t i = 0; i < len; ++i)
    if (in[a + i] != in[b + i]) return false;
  return true;
}

// The token of list entry e (stage_tokens): it starts at segment-relative byte
// r, its first 16 bytes are inside the staged buffer (bytes past the input end
// were staged as spaces), and its length, if below 16, comes with the entry.
// An inactive lane passes entry 0 and gets an empty short token: the warp takes
// one path unless a token is long.
template <class B>
__device__ __forceinline__ Tok read_token(const uint8_t* __restrict__ in, uint64_t n, uint64_t base, const B& W,
                                          uint32_t e, bool active) {
  const uint32_t* wb = reinterpret_cast<const uint32_t*>(W.buf);
  const uint32_t r = e & 0xFFFu, L = e >> 12;
  const uint32_t a = r >> 2, sh = r * 8;  // the shift counts modulo 32
  const uint32_t x0 = wb[a], x1 = wb[a + 1], x2 = wb[a + 2], x3 = wb[a + 3], x4 = wb[a + 4];
  const int bits = 8 * (int)L;
  const uint32_t u0 = low_bits(__funnelshift_r(x0, x1, sh), bits);
  const uint32_t u1 = low_bits(__funnelshift_r(x1, x2, sh), bits - 32);
  const uint32_t u2 = low_bits(__funnelshift_r(x2, x3, sh), bits - 64);
  const uint32_t u3 = low_bits(__funnelshift_r(x3, x4, sh), bits - 96) | (L << 24);
  Tok t;
  t.w0 = (uint64_t)u0 | ((uint64_t)u1 << 32);
  t.w1 = (uint64_t)u2 | ((uint64_t)u3 << 32);
  t.h = hash_short(u0, u1, u2, u3);
  if (L || !active) return t;
  // long token: FNV-1a 64 over its bytes, then the length is mixed in
  const uint64_t off = base + r;
  uint64_t h = 0xcbf29ce484222325ull, len = 0;
  for (uint64_t i = off; i < n; ++i) {
    const uint32_t rel = (uint32_t)(i - base);
    const uint32_t c = (i - base) < sizeof(W.buf) ? W.buf[rel] : in[i];
    if (is_ws(c)) break;
    h = (h ^ c) * 0x100000001b3ull;
    ++len;
  }
  t.w0 = off + 1;
  t.w1 = LONG_TAG | (len & LEN_MASK);
  t.h = (uint32_t)fmix64(h ^ len);
  return t;
}

// an even slot and the one after it (tables are 32-byte aligned)
__device__ __forceinline__ void ld_pair(const unsigned long long* p, uint64_t& a0, uint64_t& a1, uint64_t& b0,
                                        uint64_t& b1) {
  asm volatile("ld.volatile.global.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(a0), "=l"(a1), "=l"(b0), "=l"(b1)
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void cas_slot(unsigned long long* p, uint64_t n0, uint64_t n1, uint64_t& o0, uint64_t& o1) {
  asm volatile(
      "{\n\t.reg .b128 d, c, v;\n\t"
      "mov.b128 c, {%2, %2};\n\t"
      "mov.b128 v, {%3, %4};\n\t"
      "atom.relaxed.gpu.global.cas.b128 d, [%5], c, v;\n\t"
      "mov.b128 {%0, %1}, d;\n\t}\n"
      : "=l"(o0), "=l"(o1)
      : "l"(0ull), "l"(n0), "l"(n1), "l"(p)
      : "memory");
}

__device__ __forceinline__ uint64_t global_slot(uint32_t h, uint32_t log2cap) {
  return log2cap ? (uint64_t)((h * 0x9E3779B1u) >> (32 - log2cap)) : 0;
}

// Combine (key, c) into the job's global container.  Linear probing from the
// first slot of the key's pair, a pair per step with one 32-byte load (as two
// 16-byte loads the lanes' separate lines took the L1 twice as long: 4 us of 414
// for 256 MB of 50,000 words).
// Both slots are loaded before either is examined; a slot loaded before a CAS
// on the slot before it may be stale, which is harmless: a slot only ever
// changes from empty to a key.
__device__ __forceinline__ bool slot_take(const JobDev& J, uint64_t s, uint64_t r0, uint64_t r1, uint64_t w0,
                                          uint64_t w1, bool is_long, uint64_t c) {
  unsigned long long* sp = J.key + 2 * s;
  if (r0 == 0 || r1 == 0) {  // empty, or a read that raced the CAS: ask the CAS
    cas_slot(sp, w0, w1, r0, r1);
    if (r0 == 0 && r1 == 0) {
      atomicAdd(J.cnt + s, (unsigned long long)c);
      return true;
    }
  }
  if (r1 == w1 && (r0 == w0 || (is_long && long_equal(J.in, r0 - 1, w0 - 1, w1 & LEN_MASK)))) {
    atomicAdd(J.cnt + s, (unsigned long long)c);
    return true;
  }
  return false;
}

__device__ inline void global_insert(const JobDev& J, uint64_t w0, uint64_t w1, uint32_t h, uint64_t c) {
  uint64_t slot = global_slot(h, J.log2cap) & ~1ull;
  const bool is_long = (w1 >> 56) == 0xFF;
  const uint64_t mask = J.cap - 1;
  for (int p = 0; p < MAX_PROBES; p += 2) {
    uint64_t a0, a1, b0, b1;
    ld_pair(J.key + 2 * slot, a0, a1, b0, b1);
    if (slot_take(J, slot, a0, a1, w0, w1, is_long, c)) return;
    if (slot_take(J, slot + 1, b0, b1, w0, w1, is_long, c)) return;
    slot = (slot + 2) & mask;
  }
  atomicOr(J.state, 1u);
}

// Combine one token per active lane into the warp's cache; all 32 lanes call
// this together (the warp syncs inside).  A short key that sits in one of its
// two cache slots adds 1 there.  Otherwise the first of its slots that is
// empty is claimed by a CAS on the slot's w1: the winner fills the slot with
// count 1; a loser whose key turns out to be the winner's (read after a warp
// sync) adds 1 to it.  Returns true for a token the cache did not take —
// long keys (>= 16 bytes), keys whose slots are held by other keys, lost
// claims for other keys — which the caller sends to the global container.
__device__ __forceinline__ bool combine_local(WarpLocal& L, bool active, const Tok& t) {
  const bool is_long = (t.w1 >> 56) == 0xFF;
  const int s0 = (int)(t.h & (LT - 1)), s1 = (int)((t.h >> 16) & (LT - 1));
  bool done = !active;
  int want = -1;
  if (active && !is_long) {
    const uint64_t a1 = L.w1[s0], b1 = L.w1[s1];
    if (a1 == t.w1 && L.w0[s0] == t.w0) {
      atomicAdd(&L.cnt[s0], 1u);
      done = true;
    } else if (b1 == t.w1 && L.w0[s1] == t.w0) {
      atomicAdd(&L.cnt[s1], 1u);
      done = true;
    } else if (a1 == 0) {
      want = s0;
    } else if (b1 == 0) {
      want = s1;
    }
  }
  __syncwarp();
  unsigned long long old = ~0ull;
  if (want >= 0) old = atomicCAS(&L.w1[want], 0ull, (unsigned long long)t.w1);
  const bool won = want >= 0 && old == 0;
  if (won) {
    L.w0[want] = t.w0;
    L.h[want] = t.h;
    L.cnt[want] = 1u;
    done = true;
  }
  __syncwarp();
  if (want >= 0 && !won && old == t.w1 && L.w0[want] == t.w0) {
    atomicAdd(&L.cnt[want], 1u);
    done = true;
  }
  return !done;
}

__device__ inline void local_clear(WarpLocal& L) {
  for (int s = threadIdx.x & 31; s < LT; s += 32) L.w1[s] = 0;
  __syncwarp();
}

// Merge the warp's cache into the global container and empty it.
__device__ inline void local_flush(WarpLocal& L, int& occ, const JobDev& J) {
  __syncwarp();
  for (int s = threadIdx.x & 31; s < LT; s += 32) {
    if (L.w1[s] != 0) {
      global_insert(J, L.w0[s], L.w1[s], L.h[s], L.cnt[s]);
      L.w1[s] = 0;
    }
  }
  __syncwarp();
  occ = 0;
}

__device__ __forceinline__ uint4 shfl_down_u4(const uint4& v, int d) {
  return make_uint4(__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d),
                    __shfl_down_sync(0xffffffffu, v.z, d), __shfl_down_sync(0xffffffffu, v.w, d));
}
__device__ __forceinline__ uint4 shfl_u4(const uint4& v, int src) {
  return make_uint4(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src),
                    __shfl_sync(0xffffffffu, v.z, src), __shfl_sync(0xffffffffu, v.w, src));
}
// Bytes [sh, sh + 16) of the 32-byte little-endian window a | b (sh < 16).
__device__ __forceinline__ uint4 shift_window(const uint4& a, const uint4& b, uint32_t sh) {
  const uint32_t q = sh >> 2, r = (sh & 3) * 8;
  // t_i = word i + q of the window, picked without indexing registers
  const uint32_t t0 = q == 0 ? a.x : q == 1 ? a.y : q == 2 ? a.z : a.w;
  const uint32_t t1 = q == 0 ? a.y : q == 1 ? a.z : q == 2 ? a.w : b.x;
  const uint32_t t2 = q == 0 ? a.z : q == 1 ? a.w : q == 2 ? b.x : b.y;
  const uint32_t t3 = q == 0 ? a.w : q == 1 ? b.x : q == 2 ? b.y : b.z;
  const uint32_t t4 = q == 0 ? b.x : q == 1 ? b.y : q == 2 ? b.z : b.w;
  return make_uint4(__funnelshift_r(t0, t1, r), __funnelshift_r(t1, t2, r), __funnelshift_r(t2, t3, r),
                    __funnelshift_r(t3, t4, r));
}

// Stage the segment that starts at byte base (32 * B::LANE bytes, and a halo)
// in the warp's buffer W (members buf, starts), and list the tokens whose first
// byte lies in it: first byte (segment-relative) | length << 12.  A token's
// length comes from the whitespace bits of its lane and of the next one, so the
// round that reads the token needs no bitmap (eight instructions and two
// shared-memory loads less per token).  Returns how many there are.  All 32
// lanes call this.
// end: tokens that start there or beyond are left to another caller.
// The loads are not issued a segment ahead: the 24 to 32 warps of an SM hide
// them, and with the next segment's data held in registers the kernels were
// slower (256 MB 419 against 414 us, a batch of 60 jobs 640 against 621).
template <class B>
__device__ inline int stage_tokens(const JobDev& J, uint64_t base, B& L, uint64_t end = ~0ull) {
  constexpr int NCH = B::LANE / 16;  // 16-byte chunks per lane: chunk 32 c + lane
  constexpr uint32_t SB = 32 * B::LANE, BUF = SB + HALO;
  static_assert((NCH == 1 || NCH == 2) && HALO == 32 && sizeof(L.buf) == BUF, "segment layout");
  const int lane = threadIdx.x & 31;
  const uint8_t* __restrict__ in = J.in;
  const uint64_t rem = J.n - base;
  // stage the segment and its halo; bytes past the input end read as spaces
  const uintptr_t sa = reinterpret_cast<uintptr_t>(in + base);
  uint4* buf = reinterpret_cast<uint4*>(L.buf);
  uint4 ch[NCH];
  uint32_t before = ' ';  // the byte before the segment (lane 0)
  if (lane == 0 && base) before = in[base - 1];
  if (rem >= BUF && (sa & 15) == 0) {
    const uint4* src = reinterpret_cast<const uint4*>(sa);
#pragma unroll
    for (int c = 0; c < NCH; ++c) buf[32 * c + lane] = ch[c] = __ldg(src + 32 * c + lane);
    if (lane < HALO / 16) buf[32 * NCH + lane] = __ldg(src + 32 * NCH + lane);
  } else if (rem >= BUF) {
    // unaligned input: the aligned words covering the staged bytes (each
    // holds at least one input byte, so no load leaves the input's 16-byte
    // blocks), shifted into place; chunk q needs words q and q + 1
    const uint32_t sh = (uint32_t)(sa & 15);
    const uint4* src = reinterpret_cast<const uint4*>(sa - sh);
    uint4 a[NCH + 1];
#pragma unroll
    for (int c = 0; c < NCH; ++c) a[c] = __ldg(src + 32 * c + lane);
    a[NCH] = lane <= HALO / 16 ? __ldg(src + 32 * NCH + lane) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      uint4 b = shfl_down_u4(a[c], 1);
      const uint4 nx = shfl_u4(a[c + 1], 0);
      if (lane == 31) b = nx;
      buf[32 * c + lane] = ch[c] = shift_window(a[c], b, sh);
    }
    const uint4 en = shfl_down_u4(a[NCH], 1);
    if (lane < HALO / 16) buf[32 * NCH + lane] = shift_window(a[NCH], en, sh);
  } else {
    for (uint32_t r = lane; r < BUF; r += 32) L.buf[r] = r < rem ? in[base + r] : (uint8_t)' ';
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NCH; ++c) ch[c] = buf[32 * c + lane];
  }
  // whitespace bits of this lane's B::LANE consecutive bytes (ws) and of the
  // bytes after them (next)
  uint32_t ws = ws_bits(ch[0]), next;
  if (NCH == 2) {
    const uint32_t p = ws | (ws_bits(ch[NCH - 1]) << 16);
    const uint32_t p0 = __shfl_sync(0xffffffffu, p, 2 * lane), p1 = __shfl_sync(0xffffffffu, p, 2 * lane + 1);
    ws = __byte_perm(p0, p1, lane < 16 ? 0x5410 : 0x7632);
  }
  __syncwarp();  // lanes 0 and 1 staged the halo
  const uint32_t halo = __ballot_sync(0xffffffffu, is_ws(L.buf[SB + lane]));
  next = __shfl_down_sync(0xffffffffu, ws, 1);
  if (lane == 31) next = halo;
  const uint32_t last = __ballot_sync(0xffffffffu, ws >> (B::LANE - 1));
  const uint32_t first = __shfl_sync(0xffffffffu, (uint32_t)is_ws(before), 0);
  const uint32_t prev = (((last << 1) | first) >> lane) & 1u;
  uint32_t start = ~ws & ((ws << 1) | prev);
  if (NCH == 1) {
    start &= 0xFFFFu;
    ws |= next << 16;
  }
  if (base + SB > end) start = low_bits(start, (int)(end - base) - lane * B::LANE);
  const int c = __popc(start);
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  {
    uint16_t* o = L.starts + (incl - c);
    uint32_t m = start;
    while (m) {
      const uint32_t j = __ffs(m) - 1;
      // the whitespace after byte j, 15 bytes of it
      const uint32_t after = NCH == 1 ? ws >> (j + 1) : __funnelshift_rc(ws, next, j + 1);
      *o++ = (uint16_t)((lane * B::LANE + j) | (__ffs(after & 0x7FFFu) << 12));
      m &= m - 1;
    }
  }
  __syncwarp();
  return total;
}

// One warp maps and combines the tokens whose first byte lies in segment seg.
// miss(lane_has_miss, token) is called by all 32 lanes after each round of
// up to 32 tokens and disposes of the tokens the cache did not take.
template <class Miss>
__device__ inline void warp_segment_t(const JobDev& J, uint64_t seg, WarpLocal& L, int& occ, Miss&& miss) {
  const int lane = threadIdx.x & 31;
  const uint64_t base = seg * SEG;
  const int total = stage_tokens(J, base, L);
  for (int r0 = 0; r0 < total; r0 += 32) {
    const int i = r0 + lane;
    const bool active = i < total;
    Tok t;
    t = read_token(J.in, J.n, base, L, active ? L.starts[i] : 0u, active);
    const bool m = combine_local(L, active, t);
    miss(m, t);
    __syncwarp();
  }
  // occ counts segments since the last cache merge
  if (++occ >= CACHE_EPOCH) local_flush(L, occ, J);
}

// ---------------------------------------------------------------------------
// Local container of the plain map kernel for large inputs: one table per CTA
// in shared memory, shared by its warps (the paper's bounded local table,
// Sec. III-D, here per thread block).  Buckets of four slots; a slot is claimed
// once and never changes key, so once a CTA has seen a few thousand distinct
// keys the table is read-only apart from its counts, and it holds the keys that
// were frequent early on (for a Zipf-like stream, the hot ones).
//
// A bucket's word of four 8-bit tags (of the hash; 0: empty) says which slot to
// compare, so a token costs one 4-byte load and, if a tag matches, one 16-byte
// load of that slot's key; most misses load no key at all.  (Two slots' keys in
// turn, without tags, took 128 of the 360 us the map kernel spends on 256 MB of
// 50,000 words; with tags a fifth less.)  A claim CASes the tag into the word and then
// stores the key with one 16-byte store.  A slot holds w0 with 0x20 exclusive-ored
// into every byte: no token has eight spaces there, so a stored first half is
// never zero (nor is w1), and a read that meets a claim half done, where a half is
// still zero, does not match; that token, like one whose tag matches another
// key's, goes on as a miss.  (Keys whose w0 is zero, tokens of NUL bytes, were
// kept out of the table instead: 16 MiB of such tokens, all misses for one slot of
// the global container, took 9.0 ms, now 0.10.)  A key may end up in two slots (two lanes
// claiming it at once) or also in the global container, which merges them.
template <int NS>
struct CtaTableT {
  static constexpr int SLOTS = NS;  // a multiple of 4
  ulonglong2 key[NS];  // {w0 ^ SPACES, w1}; zero: empty
  uint32_t cnt[NS];
  uint32_t tag[NS / 4];
  // all threads of the CTA
  __device__ void clear() {
    for (int i = threadIdx.x; i < NS; i += blockDim.x) {
      key[i] = make_ulonglong2(0ull, 0ull);
      cnt[i] = 0;
      if (i < NS / 4) tag[i] = 0;
    }
  }
};
// the table of the large-input map kernel and the batch kernel (one CTA of
// 32 warps per SM)
using CtaTableBig = CtaTableT<4096>;

// Per-warp state beside such a table: the staged segment, its token list, and a
// queue of the tokens the table did not take, which go to the global container
// 32 at a time (full warps, so the global probing runs once per 32 misses
// instead of once per round).  With 32 bytes a lane the segment's fixed work
// (halo, scan) serves twice the tokens of 16, and the last round of up to 32
// tokens is one in four or five instead of one in two or three (256 MB of
// 50,000 words: 434 against 470 us).
constexpr int MQ = 64;
struct MapWarp {
  static constexpr int LANE = 32;  // bytes of the segment per lane
  uint8_t buf[32 * LANE + HALO];
  uint16_t starts[16 * LANE];
  unsigned long long qw0[MQ], qw1[MQ];
  uint32_t qh[MQ];
};
static_assert(sizeof(CtaTableBig) % 16 == 0 && sizeof(MapWarp) % 16 == 0, "staging buffers must stay 16-byte aligned");

constexpr uint64_t SPACES = 0x2020202020202020ull;

// Merge one slot of such a table (all keys are short) into the global container.
__device__ __forceinline__ void cta_merge(const JobDev& J, const ulonglong2& k, uint32_t c) {
  if (k.y == 0) return;
  const uint64_t w0 = k.x ^ SPACES;
  global_insert(J, w0, k.y, hash_short((uint32_t)w0, (uint32_t)(w0 >> 32), (uint32_t)k.y, (uint32_t)(k.y >> 32)), c);
}

// 0x80 in the zero bytes of v: exact up to and including the lowest one
__device__ __forceinline__ uint32_t zero_bytes(uint32_t v) { return (v - 0x01010101u) & ~v & 0x80808080u; }

// Count one token in the CTA table; false if it is long, or its bucket neither
// holds it nor has a slot that could be claimed for it.
template <class TT>
__device__ __forceinline__ bool cta_add(TT& T, const Tok& t) {
  const bool able = (t.w1 >> 56) != 0xFF;
  const uint64_t w0 = t.w0 ^ SPACES;
  const uint32_t b = __umulhi(t.h, TT::SLOTS / 4);
  const uint32_t tag = max(t.h & 0xFFu, 1u);
  const uint32_t tw = *reinterpret_cast<volatile uint32_t*>(&T.tag[b]);
  const uint32_t z = able ? zero_bytes(tw ^ (tag * 0x01010101u)) : 0u;
  bool hit = false;
  if (z) {
    const uint32_t s = 4 * b + (31 - __clz(z & -z)) / 8;
    unsigned long long k0, k1;
    asm volatile("ld.volatile.shared::cta.v2.u64 {%0, %1}, [%2];"
                 : "=l"(k0), "=l"(k1)
                 : "r"((uint32_t)__cvta_generic_to_shared(&T.key[s]))
                 : "memory");
    hit = k1 == t.w1 && k0 == w0;
    if (hit) atomicAdd(&T.cnt[s], 1u);
  }
  if (able && z == 0) {
    const uint32_t e = zero_bytes(tw);
    if (e) {
      const uint32_t q = (31 - __clz(e & -e)) / 8, s = 4 * b + q;
      hit = atomicCAS(&T.tag[b], tw, tw | (tag << (8 * q))) == tw;
      if (hit) {
        asm volatile("st.volatile.shared::cta.v2.u64 [%0], {%1, %2};" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&T.key[s])),
                     "l"(w0), "l"(t.w1)
                     : "memory");
        atomicAdd(&T.cnt[s], 1u);
      }
    }
  }
  return hit;
}

// A warp's queue of misses: once 32 are queued, the warp inserts the oldest 32
// into the global container (loading their slots a round ahead took longer: 434
// against 417 us for 256 MB, 50,000 words).  Warp-uniform.
struct MissQueue {
  uint32_t n = 0, head = 0;  // queued entries, the oldest

  // m: this lane has a miss
  __device__ __forceinline__ void push(const JobDev& J, MapWarp& W, bool m, const Tok& t) {
    const int lane = threadIdx.x & 31;
    const unsigned mm = __ballot_sync(0xffffffffu, m);
    if (!mm) return;
    if (m) {
      const uint32_t pos = (head + n + (uint32_t)__popc(mm & ((1u << lane) - 1u))) & (MQ - 1);
      W.qw0[pos] = t.w0;
      W.qw1[pos] = t.w1;
      W.qh[pos] = t.h;
    }
    n += (uint32_t)__popc(mm);
    if (n >= 32) {
      __syncwarp();
      const uint32_t e = (head + (uint32_t)lane) & (MQ - 1);
      global_insert(J, W.qw0[e], W.qw1[e], W.qh[e], 1);
      head = (head + 32) & (MQ - 1);
      n -= 32;
    }
  }
  __device__ __forceinline__ void drain(const JobDev& J, MapWarp& W) {
    const uint32_t lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < n) {
      const uint32_t e = (head + lane) & (MQ - 1);
      global_insert(J, W.qw0[e], W.qw1[e], W.qh[e], 1);
    }
    n = head = 0;
    __syncwarp();
  }
};

// The direct form: a token the cache did not take goes straight to the
// global container.
__device__ inline void warp_segment(const JobDev& J, uint64_t seg, WarpLocal& L, int& occ) {
  warp_segment_t(J, seg, L, occ, [&](bool m, const Tok& t) {
    if (m) global_insert(J, t.w0, t.w1, t.h, 1);
  });
}

}  // namespace wc
}  // namespace mrgb
