// Device-side building blocks: counter-based RNG, inverse-CDF searches,
// fixed-order reductions and the open-addressing hash.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mad_internal.cuh"

namespace mad {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplies; the key advances by the Weyl constants between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    if (round > 0) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x;
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// The four 64-bit uniforms of diamond ell: counter (ell_lo, ell_hi, 0, blk).
struct Uniforms {
  unsigned long long u0, u1, u2, u3;
};

__device__ __forceinline__ Uniforms diamond_uniforms(unsigned long long seed,
                                                     unsigned long long ell) {
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const uint4 b0 = philox4x32_10(make_uint4((uint32_t)ell, (uint32_t)(ell >> 32), 0u, 0u), key);
  const uint4 b1 = philox4x32_10(make_uint4((uint32_t)ell, (uint32_t)(ell >> 32), 0u, 1u), key);
  Uniforms u;
  u.u0 = ((unsigned long long)b0.y << 32) | b0.x;
  u.u1 = ((unsigned long long)b0.w << 32) | b0.z;
  u.u2 = ((unsigned long long)b1.y << 32) | b1.x;
  u.u3 = ((unsigned long long)b1.w << 32) | b1.z;
  return u;
}

// Uniforms of Philox blocks 2 and 3 of diamond ell: the segment-level
// uniforms of two-level alias draws (index q of (i, k, j, k') takes u_q of
// diamond_uniforms first and the q-th of these second).
__device__ __forceinline__ Uniforms alias_uniforms(unsigned long long seed, unsigned long long ell) {
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const uint4 b2 = philox4x32_10(make_uint4((uint32_t)ell, (uint32_t)(ell >> 32), 0u, 2u), key);
  const uint4 b3 = philox4x32_10(make_uint4((uint32_t)ell, (uint32_t)(ell >> 32), 0u, 3u), key);
  Uniforms u;
  u.u0 = ((unsigned long long)b2.y << 32) | b2.x;
  u.u1 = ((unsigned long long)b2.w << 32) | b2.z;
  u.u2 = ((unsigned long long)b3.y << 32) | b3.x;
  u.u3 = ((unsigned long long)b3.w << 32) | b3.z;
  return u;
}

// floor(u * total / 2^64).
__device__ __forceinline__ unsigned long long draw_target(unsigned long long u,
                                                          unsigned long long total) {
  return __umul64hi(u, total);
}

// The same for a 32-bit total: two multiplies instead of the 64 x 64-bit one's.
__device__ __forceinline__ uint32_t draw_target32(unsigned long long u, uint32_t total) {
  const unsigned long long hi = (u >> 32) * total + __umulhi((uint32_t)u, total);
  return (uint32_t)(hi >> 32);
}

// First position p in [0, len) with prefix[p] > target (masking the sign
// bit of row tables).  Clamped to len-1 when the table is inconsistent.
__device__ __forceinline__ int64_t search_u64(const uint64_t* __restrict__ prefix, int64_t len,
                                              unsigned long long target, bool* bad) {
  int64_t lo = 0, hi = len;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (__ldg((const unsigned long long*)prefix + mid) > target)
      hi = mid;
    else
      lo = mid + 1;
  }
  if (lo >= len) {
    *bad = true;
    lo = len - 1;
  }
  return lo;
}

__device__ __forceinline__ int64_t search_u32(const uint32_t* __restrict__ prefix, int64_t len,
                                              uint32_t target, uint32_t mask, bool* bad) {
  // Row lengths are below 2^31: 32-bit indices.
  int lo = 0, hi = (int)len;
  while (lo < hi) {
    const int mid = (int)(((unsigned)lo + (unsigned)hi) >> 1);
    if ((__ldg(prefix + mid) & mask) > target)
      hi = mid;
    else
      lo = mid + 1;
  }
  if (lo >= (int)len) {
    *bad = true;
    lo = (int)len - 1;
  }
  return lo;
}

// Branch-free upper bound with a fixed number of steps (floor(log2 len) +
// 1, the same for every lane of a row length): the number of entries <=
// target, i.e. the position of the first entry above it.
__device__ __forceinline__ int ub_steps(int len) { return 32 - __clz(len); }

__device__ __forceinline__ int ub_u32(const uint32_t* __restrict__ P, int len, uint32_t target,
                                      uint32_t mask) {
  int pos = 0;
  for (int step = 1 << (31 - __clz(len)); step > 0; step >>= 1) {
    const int np = pos + step;
    const uint32_t v = __ldg(P + (np <= len ? np : len) - 1) & mask;
    pos = (np <= len && v <= target) ? np : pos;
  }
  return pos;
}

// Upper bound in a long row through its guide: bucket b = target >> sh
// holds the answer between guide entries b and b + 1, and the prefix
// entries between those positions are counted (a window of 4, else of 16,
// else a binary search over the bucket's range).  Same result as ub_u32
// over the whole row.
__device__ __forceinline__ int ub_guided_u32(const uint32_t* __restrict__ P,
                                             const uint32_t* __restrict__ G, int sh,
                                             uint32_t target, uint32_t mask = 0xFFFFFFFFu) {
  const uint32_t b = target >> sh;
  const int lo = (int)__ldg(G + b), hi = (int)__ldg(G + b + 1);
  if (hi - lo <= 4) {
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = lo + q;
      if (e < hi) cnt += ((__ldg(P + e) & mask) <= target) ? 1 : 0;
    }
    return lo + cnt;
  }
  if (hi - lo <= 16) {
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int e = lo + q;
      if (e < hi) cnt += ((__ldg(P + e) & mask) <= target) ? 1 : 0;
    }
    return lo + cnt;
  }
  return lo + ub_u32(P + lo, hi - lo, target, mask);
}

// The same for a 64-bit prefix (T1): bucket b = target >> sh.
__device__ __forceinline__ int64_t ub_guided_u64(const uint64_t* __restrict__ P, int64_t len,
                                                 const uint32_t* __restrict__ G, int sh,
                                                 unsigned long long target) {
  const unsigned long long b = target >> sh;
  const int64_t lo = (int64_t)__ldg(G + b), hi = (int64_t)__ldg(G + b + 1);
  if (hi - lo <= 4) {
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t e = lo + q;
      if (e < hi) cnt += (__ldg(P + e) <= target) ? 1 : 0;
    }
    return lo + cnt;
  }
  if (hi - lo <= 16) {
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int64_t e = lo + q;
      if (e < hi) cnt += (__ldg(P + e) <= target) ? 1 : 0;
    }
    return lo + cnt;
  }
  int64_t pos = lo, n = hi - lo;   // first entry above target in [lo, hi)
  while (n > 0) {
    const int64_t half = n >> 1;
    if (__ldg(P + pos + half) <= target) {
      pos += half + 1;
      n -= half + 1;
    } else {
      n = half;
    }
  }
  return pos < len ? pos : len;
}

// FP32 sums of products against the exact c (d <= 1024, 32 lane partials
// folded in halves): |c~ - c| <= kBoundEps sum |a_k b_k| + kBoundTiny (the
// derivation stands with k_rescore_bound).
constexpr float kBoundEps = 1.02f * 64.0f / 16777216.0f;
constexpr float kBoundTiny = 1e-37f;

// Bits of x (0 for 0).
__device__ __forceinline__ int bitlen_u32(uint32_t x) { return x ? 32 - __clz(x) : 0; }

// Bucket shift of the guide of a 0/1 T2 row of len >= kGuideMin entries and
// total tot: the smallest that leaves at most about len / 2 buckets (with len /
// 4 the 0/1 sampler took 4.69 instead of 4.62 ms on 1e6 nodes, with len 4.63).
__device__ __forceinline__ int t2_guide_shift(uint32_t len, uint32_t tot) {
  const int sh = bitlen_u32(tot - 1) - bitlen_u32(len / 4);
  return sh > 0 ? sh : 0;
}

// Two searches over rows of the same length at once (independent loads).
__device__ __forceinline__ void ub2_u32(const uint32_t* __restrict__ P, const uint32_t* __restrict__ Q,
                                        int len, uint32_t tp, uint32_t tq, uint32_t mask, int* op,
                                        int* oq) {
  int a = 0, b = 0;
  for (int step = 1 << (31 - __clz(len)); step > 0; step >>= 1) {
    const int na = a + step, nb = b + step;
    const uint32_t va = __ldg(P + (na <= len ? na : len) - 1) & mask;
    const uint32_t vb = __ldg(Q + (nb <= len ? nb : len) - 1) & mask;
    a = (na <= len && va <= tp) ? na : a;
    b = (nb <= len && vb <= tq) ? nb : b;
  }
  *op = a;
  *oq = b;
}

// ---- TB in 64-byte blocks ----------------------------------------------------
// The draw of j is one aligned 64-byte read.  Row k's targets [0, total) are
// cut into about n / kBlockKeys equal buckets, bucket of target t = t * mul /
// 2^32; block b holds lo, the number of the row's entries at most bucket b's
// first target, and entries lo, lo + 1, ... up to 15 of them (sign bits
// included), padded with entries above every target.  The first entry above
// a target of the bucket is among entries lo .. lo', lo' the next block's lo, so
// it is in the block when lo' - lo < 15 (all but 0.1 % of the buckets where
// six entries a bucket are expected); otherwise TB is searched between the two.
// Against the row guides of tb_guide_build (two entries of the guide, then a
// window of up to 17 entries of TB at any alignment: three or four 64-byte
// fetches from DRAM for a million items, 383 bytes a diamond with b_k'j) this
// is one, for 10.7 bytes an entry of TB instead of at most 4: 1e4 queries of 5e4
// diamonds, draws 38.3 -> 29.1 ms.

// First target of bucket b: the smallest t with t * mul >= b * 2^32.
__device__ __forceinline__ unsigned long long bucket_first(unsigned long long b,
                                                           unsigned long long mul) {
  return ((b << 32) + mul - 1) / mul;
}

// First entry of row k of TB above target and its sign bit, for the 32 draws of
// a warp (all lanes).  Four lanes read a block together, eight blocks to an
// instruction: random reads from DRAM are limited by their number (3.9e10 a second
// over 4.4 GB, of 32 or of 64 bytes alike), and a block read by one lane in
// four loads is two of them, one per sector: draws of
// 5e8 diamonds on 1e6 items 27.9 ms, 22.0 so.
__device__ __forceinline__ int64_t ub_block(const SampleParams& p, int64_t nb, int64_t k,
                                            uint32_t mul, uint32_t target, uint32_t* sign) {
  const uint32_t lane = threadIdx.x & 31u, piece = lane & 3u;
  const uint32_t at = (uint32_t)(k * (nb + 1)) + __umulhi(target, mul);
  uint4 w[4];
  uint32_t tg[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {   // the blocks of lanes 8 r .. 8 r + 7
    const uint32_t b = __shfl_sync(0xFFFFFFFFu, at, 8 * r + (lane >> 2));
    tg[r] = __shfl_sync(0xFFFFFFFFu, target, 8 * r + (lane >> 2));
    w[r] = __ldg(p.tb_blocks + (size_t)b * 4 + piece);
  }
  uint32_t first = 0, head = 0;   // of this lane's block: word << 1 | sign, lo
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint32_t v[4] = {w[r].x, w[r].y, w[r].z, w[r].w};
    uint32_t f = 32u;   // first word above the target: the smallest over the four lanes
#pragma unroll
    for (int c = 3; c >= 0; --c)
      if ((c > 0 || piece > 0) && (v[c] & PREFIX_MASK) > tg[r])
        f = (piece * 4 + c) << 1 | v[c] >> 31;
    f = min(f, __shfl_xor_sync(0xFFFFFFFFu, f, 1));
    f = min(f, __shfl_xor_sync(0xFFFFFFFFu, f, 2));
    f = __shfl_sync(0xFFFFFFFFu, f, 4 * (lane & 7u));
    const uint32_t h = __shfl_sync(0xFFFFFFFFu, v[0], 4 * (lane & 7u));
    if ((lane >> 3) == (uint32_t)r) {
      first = f;
      head = h;
    }
  }
  *sign = first << 31;
  if (first < 32u) return (int64_t)head + (first >> 1) - 1;
  // Every entry held is at most the target: search on to the next block's lo.
  const uint32_t* __restrict__ row = p.TB + k * p.n;
  const uint32_t lo = head + kBlockEnts;
  const uint32_t hi = __ldg((const uint32_t*)(p.tb_blocks + ((size_t)at + 1) * 4));
  const int64_t j =
      (int64_t)lo + (hi > lo ? ub_u32(row + lo, (int)(hi - lo), target, PREFIX_MASK) : 0);
  if (j < p.n) *sign = __ldg(row + j) & SIGN_BIT;
  return j;
}

// A length known only on the device: min(cap, *n_dev), or cap itself when
// there is no device count.
__device__ __forceinline__ unsigned long long dev_len(unsigned long long cap,
                                                      const unsigned long long* n_dev) {
  if (!n_dev) return cap;
  const unsigned long long n = *n_dev;
  return n < cap ? n : cap;
}

// 2^e as an FP32 value, -126 <= e <= 127.
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// b * 2^F rounded to the nearest integer, ties to even, as int64 (callers
// keep |b * 2^F| < 2^63).  Scaling an FP32 value by a power of two is exact
// while the product stays a normal number, so the product is formed exactly
// (in two steps when 2^F itself is outside the normal range, each step
// keeping its result normal) and converted once with round-to-nearest-even.
// A product below 2^-126 in magnitude rounds to 0 whatever its last bits.
__device__ __forceinline__ long long fixed_point(float b, int F) {
  float x;
  if (F > 127) {
    x = (b * pow2f(127)) * pow2f(min(F - 127, 127));
  } else if (F < -126) {
    x = (b * pow2f(-126)) * pow2f(max(F + 126, -126));
  } else {
    x = b * pow2f(F);
  }
  return __float2ll_rn(x);
}

// Sorted-list membership (0/1 CSR closure test).
__device__ __forceinline__ bool contains_sorted(const int32_t* __restrict__ list, int64_t len,
                                                int32_t value) {
  int64_t lo = 0, hi = len;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    const int32_t v = __ldg(list + mid);
    if (v < value)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo < len && __ldg(list + lo) == value;
}

// Exponent of a positive finite FP32 value (floor(log2 x)), from its bits.
__device__ __forceinline__ int ilogb_pos(float x) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xFF);
  if (e != 0) return e - 127;
  // subnormal: value = mantissa * 2^-149
  const uint32_t mant = b & 0x7FFFFF;
  return (31 - __clz(mant)) - 149;
}

// 2^e as a double, for |e| <= 1022.
__device__ __forceinline__ double pow2d(int e) {
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// ---------------------------------------------------------------------------
// Open-addressing hash for X: 64-bit keys (EMPTY_KEY = free), int64 values,
// linear probing from a splitmix64-finalised slot.
// ---------------------------------------------------------------------------
// 32-bit finaliser of MurmurHash3 (Appleby): spreads a column index over a
// home region (the row is fixed within a region, so the column suffices).
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
  h ^= h >> 16;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return h;
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Linear probing from `slot`, wrapping at cap, four slots per round trip:
// the keys of the 32-byte group holding `slot` are read with two 16-byte
// loads, and the first slot of the group (from `slot` on) that is empty or
// holds the key is picked without branching (lanes of a warp stay
// converged).  A key already there gets the value added; an empty slot is
// claimed with one CAS, and a CAS lost to another key re-reads the group
// from that slot, so slots are still taken in linear-probing order.
// Probing wraps from slot hi back to slot lo ([lo, hi) is the whole table,
// or a region whose bounds are multiples of 4).  Returns 0 when the probe
// limit is hit, 1 when the key existed, 2 when this call created it.
__device__ __forceinline__ int hash_add_from(unsigned long long* __restrict__ keys,
                                             long long* __restrict__ vals, uint64_t lo,
                                             uint64_t hi, uint64_t slot, uint32_t max_probe,
                                             unsigned long long key, long long v) {
  uint32_t probes = 0;
  while (probes < max_probe) {
    const uint64_t g = slot & ~3ull;
    // Slots of the group at or past hi (a table size that is not a multiple
    // of 4) are skipped; probing wraps to slot lo after the group.
    const uint32_t valid = (g + 4 <= hi) ? 4u : (uint32_t)(hi - g);
    unsigned long long k4[4];
    if (valid == 4) {
      // L2 loads: keys only ever change from EMPTY to a key, and a stale
      // EMPTY is caught by the CAS.
      const ulonglong2 a = __ldcg((const ulonglong2*)(keys + g));
      const ulonglong2 b = __ldcg((const ulonglong2*)(keys + g + 2));
      k4[0] = a.x; k4[1] = a.y; k4[2] = b.x; k4[3] = b.y;
    } else {
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q) k4[q] = (q < valid) ? __ldcg(keys + g + q) : 0ull;
    }
    const uint32_t start = (uint32_t)(slot - g);
    uint32_t pick = 4;
#pragma unroll
    for (int q = 3; q >= 0; --q) {
      const bool usable = (uint32_t)q >= start && (uint32_t)q < valid &&
                          (k4[q] == key || k4[q] == EMPTY_KEY);
      pick = usable ? (uint32_t)q : pick;
    }
    if (pick == 4) {
      probes += valid > start ? valid - start : 0u;
      slot = g + 4;
      if (slot >= hi) slot = lo;
      continue;
    }
    probes += pick - start + 1;
    unsigned long long cur = k4[0];
#pragma unroll
    for (uint32_t q = 1; q < 4; ++q) cur = (q == pick) ? k4[q] : cur;
    int created = 0;
    if (cur != key) {
      const unsigned long long prev = atomicCAS(keys + g + pick, EMPTY_KEY, key);
      if (prev != EMPTY_KEY && prev != key) {
        slot = g + pick;  // taken by another key: look again from here
        --probes;         // (counted again there)
        continue;
      }
      created = prev == EMPTY_KEY ? 2 : 0;
    }
    atomicAdd((unsigned long long*)vals + g + pick, (unsigned long long)v);
    return created ? 2 : 1;
  }
  return 0;
}

// Log buckets of positive 64-bit values: 16 * floor(log2 v) + the 4 bits
// below the leading bit (1024 buckets, monotone in v), and a bucket's
// smallest value.
__device__ __forceinline__ uint32_t log_bucket(unsigned long long v) {
  const int e = 63 - __clzll((long long)v);
  const uint32_t f = e >= 4 ? (uint32_t)(v >> (e - 4)) & 15u : (uint32_t)(v << (4 - e)) & 15u;
  return (uint32_t)e * 16u + f;
}

__host__ __device__ __forceinline__ unsigned long long bucket_floor(uint32_t b) {
  const int e = (int)(b >> 4);
  const unsigned long long m = 16ull + (b & 15u);
  return e >= 4 ? (m << (e - 4)) : (m >> (4 - e));
}

// Bloom filter for the 0/1 closure test: the entry (a, b) sets five bits in
// one 64-bit word, two in its low half and three in its high half.  Word and
// bits come from two 32-bit mixes of the pair, its halves first spread by 2^32
// over the golden ratio and two of xxHash32's primes (Collet) (a 64-bit mix of the pair and a
// second one for the bits took about a fifth of the sampler's instructions).
// A clear bit proves the entry absent; a set filter sends the test to the
// exact search.
struct BloomProbe {
  unsigned long long word;
  uint32_t lo, hi;
};

__device__ __forceinline__ BloomProbe bloom_probe(uint32_t a, uint32_t b, int shift) {
  const uint32_t x = a * 0x9E3779B1u, y = b * 0x85EBCA77u;
  const uint32_t h1 = fmix32(x + y);
  const uint32_t h2 = fmix32(x ^ __funnelshift_l(y, y, 13) ^ 0x27D4EB2Fu);
  BloomProbe p;
  // The top bits of (h1, h2) taken as 40 bits (words of 2^10 to 2^40).
  p.word = (((unsigned long long)h1 << 8) | (h2 >> 24)) >> shift;
  p.lo = (1u << (h2 & 31u)) | (1u << ((h2 >> 5) & 31u));
  p.hi = (1u << ((h2 >> 10) & 31u)) | (1u << ((h2 >> 15) & 31u)) | (1u << ((h2 >> 20) & 31u));
  return p;
}

// kFar: the word is the first that L2 drops again.
template <bool kFar = false>
__device__ __forceinline__ bool bloom_may_contain(const unsigned long long* __restrict__ words,
                                                  int shift, uint32_t a, uint32_t b) {
  const BloomProbe p = bloom_probe(a, b, shift);
  const uint2* __restrict__ at = reinterpret_cast<const uint2*>(words) + p.word;
  uint2 w;
  if (kFar) {
    unsigned long long policy;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm("ld.global.nc.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
        : "=r"(w.x), "=r"(w.y)
        : "l"(at), "l"(policy));
  } else {
    w = __ldg(at);
  }
  return (w.x & p.lo) == p.lo && (w.y & p.hi) == p.hi;
}

// Place of column b in a home region of `size` slots (a power of two).  A region
// built whole (k_build_x) and one filled by k_insert place their keys alike, so
// that either finds what the other left.
__device__ __forceinline__ unsigned long long region_offset(uint32_t b, unsigned long long size) {
  return (size <= (1ull << 32) ? (unsigned long long)fmix32(b) : mix64(b)) & (size - 1);
}

// First slot probed for key = (a << 32) | b.
//
// The home regions are sized for the diamonds whose row i is theirs.  Under
// MAD_GRAM the key (min(i, j), max(i, j)) no longer tells which end was i: with
// the region of a as the home, low rows collected up to twice what theirs were
// sized for and high rows nothing, and probes ran through whole stretches of
// full regions (30,011 x 63 FP64, 2e6 diamonds: k_insert 1115 us, the fused
// pass 1431 us; with the homes below the pass takes 426 us).  There the
// home is the region of a or of b, by a hash of the key in proportion to the
// two sizes: for vectors of norms n_r the load of row r against its size is
// then R (R + 1) / (R^2 + 1) of the plain one with R = n_r / the mean norm,
// at most 1.21, whatever the order of the rows.
__device__ __forceinline__ uint64_t home_slot(const SampleParams& p, unsigned long long key) {
  if (p.regioned) {
    const uint32_t a = (uint32_t)(key >> 32), b = (uint32_t)key;
    unsigned long long r0 = p.hreg[a];
    unsigned long long size = p.hreg[a + 1] - r0;  // a power of two
    if (p.flags & MAD_GRAM) {
      const unsigned long long h = mix64(key);
      const unsigned long long rb = p.hreg[b];
      const unsigned long long sb = p.hreg[b + 1] - rb;
      if (__umul64hi(h, size + sb) >= size) {
        r0 = rb;
        size = sb;
      }
      return r0 + (h & (size - 1));
    }
    return r0 + region_offset(b, size);
  }
  return mix64(key) & p.hmask;
}

__device__ __forceinline__ int hash_add(const SampleParams& p, unsigned long long key, long long v) {
  return hash_add_from(p.hkeys, p.hvals, 0, p.hcap, home_slot(p, key), p.max_probe, key, v);
}

// Histogram pick by one whole block of 256 threads: the highest bucket b
// whose count from the top (buckets b .. NB-1) reaches K, or -1 when the
// total stays below K; *total receives the sum of all buckets.  The counts
// are read from global memory (L2), each thread owning NB/256 consecutive
// buckets from the top, and a block scan finds the thread whose range the
// running count crosses.  Every thread of the block must call it.
template <int NB>
__device__ int block_pick_from_top(const unsigned int* hist, unsigned long long K,
                                   unsigned long long* total) {
  static_assert(NB % 256 == 0, "buckets per thread");
  constexpr int PER = NB / 256;
  __shared__ unsigned long long csum[256];
  __shared__ int pick;
  const int t = threadIdx.x;
  unsigned int v[PER];
  unsigned long long mine = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    v[q] = __ldcg(hist + (NB - 1 - (t * PER + q)));
    mine += v[q];
  }
  csum[t] = mine;
  if (t == 0) pick = -1;
  __syncthreads();
  for (int off = 1; off < 256; off <<= 1) {
    const unsigned long long add = t >= off ? csum[t - off] : 0ull;
    __syncthreads();
    csum[t] += add;
    __syncthreads();
  }
  const unsigned long long before = t ? csum[t - 1] : 0ull;
  if (before < K && csum[t] >= K) {
    unsigned long long cum = before;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      cum += v[q];
      if (cum >= K) {
        pick = NB - 1 - (t * PER + q);
        break;
      }
    }
  }
  __syncthreads();
  *total = csum[255];
  return pick;
}

}  // namespace mad
