// The sampling loop of Alg. 2: for every diamond index l, draw the center
// edge (i,k) with probability w_ik / ||W||_1 (two stages: row i from T1,
// then k from row i of T2), j with probability |b_kj| / ||b_k*||_1 (row k of
// TB), k' with probability |a_ik'| / ||a_i*||_1 (row i of TA), and add
// sgn(a_ik b_kj a_ik') b_k'j to x_ij (Alg. 2 increment line).
//
// GPU organisation: one diamond per thread; the signs of a_ik, b_kj and
// a_ik' come for free with the table entries the searches land on (bit 31),
// so only b_k'j is read from B.  Lanes of a warp whose diamonds hit the same
// key combine their increments before one lane inserts into the hash.
//
// Dense inputs are processed in row order: a counting sort by the row i of
// each diamond's center edge (drawn from T1 alone) groups the diamonds, so
// the lanes of a warp mostly share row i and its T2/TA/A entries come from
// L1 once per row instead of once per diamond, and the hash keys (i, j) of
// the rows in flight fall into a narrow band of home regions that stays in
// L2.  The draws of every diamond are unchanged by the reordering.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "draw.cuh"
#include "mad_device.cuh"
#include "mad_internal.cuh"

namespace mad {
namespace {

// The scalars derived from T1's total on the device (and, for the dense
// hash, the end of its home regions), read once per thread, so that no
// host round trip separates the table build from the sampler.
__device__ __forceinline__ SampleParams resolve(const SampleParams& p) {
  SampleParams q = p;
  q.t1_total = p.sc->t1_total;
  q.t1g_sh = p.sc->t1g_sh;
  q.f_exp = p.sc->f_exp;
  if (p.regioned) {
    const unsigned long long used = p.hreg[p.m];
    q.hcap = used < p.hcap_alloc ? used : p.hcap_alloc;
  }
  return q;
}

// Per-lane bookkeeping of the sampling kernels.
struct Tally {
  unsigned long long inserted = 0, diag = 0, created = 0;
  bool bad = false, full = false;
};

// Filter one drawn diamond and add it to X.  Lanes holding the same key
// insert independently (the atomics combine them).
// One addition of v to the pair (a, b) (unordered under MAD_GRAM).
__device__ __forceinline__ void add_pair(const SampleParams& p, uint32_t a, uint32_t b, long long v,
                                         Tally& t) {
  if ((p.flags & MAD_EXCLUDE_DIAG) && a == b) {
    ++t.diag;
    return;
  }
  if (v == 0) return;
  if ((p.flags & MAD_GRAM) && b < a) {
    const uint32_t c = a;
    a = b;
    b = c;
  }
  ++t.inserted;
  const int r = hash_add(p, ((unsigned long long)a << 32) | b, v);
  if (r == 0) t.full = true;
  if (r == 2) ++t.created;
}

// Filter one drawn diamond and add it to X: to the pair (i, j), and under
// MAD_SQUARE_SYM also to the pair (k, k') (Sec. 3.2.3).  Lanes holding the
// same key insert independently (the atomics combine them).
__device__ __forceinline__ void accumulate(const SampleParams& p, bool valid, const Draw& dr,
                                           Tally& t) {
  if (!valid) return;
  add_pair(p, dr.i, dr.j, dr.v, t);
  if (p.flags & MAD_SQUARE_SYM) add_pair(p, dr.k, dr.kp, dr.v, t);
}

// The same, reduced over the whole block first (one atomic per counter and
// block: kernels with many short blocks would otherwise queue thousands of
// atomics on the same counters).  Every thread of the block calls it.
__device__ __forceinline__ void flush_tally_block(const SampleParams& p, Tally& t) {
  __shared__ unsigned long long s_ins, s_cre;
  __shared__ unsigned int s_flags;
  if (threadIdx.x == 0) {
    s_ins = 0;
    s_cre = 0;
    s_flags = 0;
  }
  __syncthreads();
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    t.inserted += __shfl_xor_sync(0xFFFFFFFFu, t.inserted, off);
    t.created += __shfl_xor_sync(0xFFFFFFFFu, t.created, off);
  }
  const unsigned any_full = __ballot_sync(0xFFFFFFFFu, t.full);
  if ((threadIdx.x & 31) == 0) {
    if (t.inserted) atomicAdd(&s_ins, t.inserted);
    if (t.created) atomicAdd(&s_cre, t.created);
    if (any_full) atomicOr(&s_flags, 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_ins) atomicAdd(&p.sc->inserted, s_ins);
    if (s_cre) atomicAdd(&p.sc->new_keys, s_cre);
    if (s_flags) atomicOr(&p.sc->err, DERR_HASH_FULL);
  }
}

__device__ __forceinline__ void flush_tally(const SampleParams& p, Tally& t) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    t.inserted += __shfl_xor_sync(0xFFFFFFFFu, t.inserted, off);
    t.diag += __shfl_xor_sync(0xFFFFFFFFu, t.diag, off);
    t.created += __shfl_xor_sync(0xFFFFFFFFu, t.created, off);
  }
  const unsigned any_bad = __ballot_sync(0xFFFFFFFFu, t.bad);
  const unsigned any_full = __ballot_sync(0xFFFFFFFFu, t.full);
  if (lane == 0) {
    if (t.inserted) atomicAdd(&p.sc->inserted, t.inserted);
    if (t.diag) atomicAdd(&p.sc->diag_skipped, t.diag);
    if (t.created) atomicAdd(&p.sc->new_keys, t.created);
    if (any_bad) atomicOr(&p.sc->err, DERR_SEARCH);
    if (any_full) atomicOr(&p.sc->err, DERR_HASH_FULL);
  }
}

// Diamonds in index order: dense inputs with alias draws, and 0/1 inputs whose
// indices do not fit the row descriptors (k_sample_rows takes the others).
template <bool kAlias>
__global__ void __launch_bounds__(256)
k_sample(const SampleParams p_, unsigned long long seed, unsigned long long first,
         unsigned long long s) {
  const SampleParams p = resolve(p_);
  const int lane = threadIdx.x & 31;
  const unsigned long long warp_id = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const unsigned long long warps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  Tally t;
  for (unsigned long long base = warp_id * 32; base < s; base += warps * 32) {
    const unsigned long long q = base + lane;
    Draw dr{};
    if (q < s) dr = draw_one_as<kAlias>(p, seed, first + q, &t.bad);
    accumulate(p, q < s, dr, t);
  }
  flush_tally(p, t);
}

// 0/1 inputs: the loop body of Alg. 2 with what it needs of a row in one load
// (SampleParams::rdesc, brow); the draws are those of draw_given_row.  v is 1
// where the diamond closes.  Every lane of the warp calls it.
//
// Bound by random sectors (about ten a diamond: T1's guide, the row, its guide
// and window of T2, the two columns, the row of B, its column, the filter
// word), at 54 % of DRAM's rate, 64 % of L2's and 66 % of L1's at once, so it
// wants every warp the SM holds (32 registers).  Five arrays' worth of row data
// in one 16-byte load, a cheaper filter mix and T2 guides of about four entries
// a bucket took 1e8 diamonds on the graph of 1e6 nodes from 6.12 to 4.62 ms
// (3e7 on 20,011 nodes, all in L2: 1.63 to 1.34).  Tried and dropped: the same
// diamonds in the order of their rows (the sort costs what the locality
// saves, 4.77 ms at best), windows read as 16-byte quads (registers spill,
// 7.0 ms), and leaving the loop body early where the filter rules a diamond
// out (the warp's lanes then run apart for good, 10.1 ms).
template <bool kFar>
__device__ __forceinline__ Draw draw_rows(const SampleParams& p, bool valid,
                                          unsigned long long seed, unsigned long long ell,
                                          bool* bad) {
  const bool gram = (p.flags & MAD_GRAM) != 0;
  Draw dr{};
  bool maybe = false;
  if (valid) {
    const Uniforms u = diamond_uniforms(seed, ell);
    int64_t i = ub_guided_u64(p.T1, p.m, p.T1g, p.t1g_sh, draw_target(u.u0, p.t1_total));
    if (i >= p.m) { *bad = true; i = p.m - 1; }
    const uint4 ra = __ldg(p.rdesc + i);
    const uint32_t* __restrict__ row = p.T2 + ra.x;
    const uint32_t target = draw_target32(u.u1, ra.z);
    uint32_t pk =
        ra.y >= (uint32_t)kGuideMin
            ? (uint32_t)ub_guided_u32(row, p.T2g + ra.w, t2_guide_shift(ra.y, ra.z), target)
            : (uint32_t)ub_u32(row, (int)ra.y, target, 0xFFFFFFFFu);
    if (pk >= ra.y) { *bad = true; pk = ra.y - 1; }
    const uint32_t pkp = draw_target32(u.u3, ra.y);
    dr.i = (uint32_t)i;
    dr.k = (uint32_t)__ldg(p.a_col + ra.x + pk);
    dr.kp = (uint32_t)__ldg(p.a_col + ra.x + pkp);
    const uint2 rb = __ldg(p.brow + dr.k);
    dr.j = (uint32_t)__ldg(p.b_col + rb.x + draw_target32(u.u2, rb.y));
    // b_k'j != 0: the entry (j, k') of A under MAD_GRAM, else (k', j) of B.
    maybe = !p.bloom || bloom_may_contain<kFar>(p.bloom, p.bloom_shift, gram ? dr.j : dr.kp,
                                                gram ? dr.kp : dr.j);
  }
  // The few lanes whose diamond may close are searched while the others wait,
  // and the warp goes on together.
  if (__any_sync(0xFFFFFFFFu, maybe)) {
    if (maybe) {
      const uint2 rc = __ldg(p.brow + dr.kp);
      const uint4 rj = gram ? __ldg(p.rdesc + dr.j) : make_uint4(0u, 0xFFFFFFFFu, 0u, 0u);
      // (under MAD_GRAM b_k'j = a_jk': the shorter of the two sorted rows)
      const bool hit = gram && rj.y < rc.y
                           ? contains_sorted(p.a_col + rj.x, rj.y, (int32_t)dr.kp)
                           : contains_sorted(p.b_col + rc.x, rc.y, (int32_t)dr.j);
      dr.v = hit ? 1 : 0;
    }
    __syncwarp();
  }
  return dr;
}

template <bool kFar>
__global__ void __launch_bounds__(256, 8)
k_sample_rows(const SampleParams p_, unsigned long long seed, unsigned long long first,
              unsigned long long s) {
  const SampleParams p = resolve(p_);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long rounds = (s + stride - 1) / stride;
  Tally t;
  unsigned long long x = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (unsigned long long r = 0; r < rounds; ++r, x += stride) {
    const bool valid = x < s;
    const Draw dr = draw_rows<kFar>(p, valid, seed, first + x, &t.bad);
    accumulate(p, valid, dr, t);
    __syncwarp();
  }
  flush_tally(p, t);
}

// Counting sort of diamonds into row order.  A diamond's bucket is the top
// bits of its stage-1 target (Philox block 0 and T1's total only): the row
// i = upper_bound(T1, target) is non-decreasing in the target, so bucket
// order is row order; the T1 search itself is left to the draw kernel,
// where neighbouring diamonds search the same few lines of T1.  At most
// 2^kSortBitsMax buckets (a few rows each; measured on the dense factor
// workload, 2^14 buckets made sampling 3.7 % slower than 2^15).
//
// Two levels: the top kCoarseBits of the bucket across the grid, then the rest
// inside each coarse bucket.
//  1. k_sort_scatter: a block takes a contiguous chunk of the diamonds, a tile of
//     8192 at a time: a tile is ordered by coarse bucket in shared memory, takes
//     its places in the buckets' slots with one atomic per bucket, and its records
//     (diamond index and the bucket's low bits, one word) leave in runs of about
//     eight, whole sectors.  The target is uniform, so a coarse bucket gets
//     s * width / total diamonds give or take: it has slots for that and three
//     standard deviations, and what is more goes to a list of its own (some ten of
//     1e7 diamonds).  No pass counts the diamonds first.
//  2. k_sort_fine: a block per coarse bucket orders its records by the low bits in
//     shared memory and writes indices and bucket offsets in order.
// Bound by Philox and the scatter's shared-memory steps.  One level
// over all 2^16 buckets kept a count per (bucket, block), as many as there were
// diamonds, through four passes (40 MB: 67 us of sums and offsets), and wrote
// each index to a sector of its own (94 us): 206 us with the histogram; two levels
// with a counting pass (34 us) and a scan of its counts 123; without them 89 (cold
// caches, one by one; the fused pass 965 -> 930 -> 904 with other changes -> 874 us).
constexpr int kSortBitsMax = 16;
constexpr int kCoarseBits = 10;
constexpr int kSortThreads = 1024;
constexpr int kTilePer = 8;                             // diamonds per thread and tile
constexpr int kSortTile = kSortThreads * kTilePer;
constexpr int kIdxBits = 26;                            // diamond index in a record
constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1u;
constexpr uint32_t kFineStage = 24576;                  // records k_sort_fine holds in shared memory

__device__ __forceinline__ uint32_t sort_bucket(unsigned long long ell, uint2 key,
                                                unsigned long long t1_total, int shift) {
  const uint4 b0 = philox4x32_10(make_uint4((uint32_t)ell, (uint32_t)(ell >> 32), 0u, 0u), key);
  const unsigned long long u0 = ((unsigned long long)b0.y << 32) | b0.x;
  return (uint32_t)(draw_target(u0, t1_total) >> shift);
}

// Slots of a coarse bucket (see above): the same in every block of both kernels.
// shift: of a coarse bucket; slots_max bounds them all together.
__device__ __forceinline__ uint32_t coarse_slots(unsigned long long s, unsigned long long total,
                                                 int shift, unsigned long long slots_max) {
  const double mean = (double)s * ldexp(1.0, shift) / (double)total;
  const unsigned long long used = ((total - 1) >> shift) + 1, most = slots_max / used;
  const unsigned long long want = (unsigned long long)(fmin(mean, 4e9) + 3.0 * sqrt(mean)) + 1;
  return (uint32_t)(want < most ? want : most);
}

// Exclusive scan of one value per thread over a 1024-thread block.
__device__ __forceinline__ uint32_t block_exclusive_1024(uint32_t v, uint32_t* warp_sum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = warp_sum[lane];
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += y;
    }
    warp_sum[lane] = wi - w;
  }
  __syncthreads();
  return warp_sum[warp] + inc - v;
}

struct SortTile {
  uint32_t cur[1 << kCoarseBits];    // the tile's first place in each coarse bucket
  uint32_t cnt[1 << kCoarseBits];    // this tile's counts
  uint32_t off[1 << kCoarseBits];    // their exclusive scan
  uint32_t rec[kSortTile];
  uint16_t bkt[kSortTile];
  uint32_t warp_sum[32];
  uint32_t slots;
};

// Places given out in each coarse bucket, and the length of the list of those
// beyond its slots.
struct SortTaken {
  unsigned int n[1 << kCoarseBits], over;
};

// Step 1: rec[c * slots + place] = low bucket bits << kIdxBits | q for every
// diamond q of the block's chunk, c its coarse bucket; places from slots on go to
// over instead, with c.  taken: the places given out, zero at first.
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_scatter(const DevScalars* __restrict__ sc, unsigned long long seed,
               unsigned long long first, unsigned long long s, unsigned long long chunk,
               int coarse, int fine, unsigned long long slots_max, SortTaken* taken,
               uint32_t* __restrict__ rec, uint2* __restrict__ over) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  SortTile& sh = *reinterpret_cast<SortTile*>(sort_smem);
  const int tid = threadIdx.x, nc = 1 << coarse;
  static_assert((1 << kCoarseBits) == kSortThreads, "a coarse bucket per thread");
  if (tid == 0) sh.slots = coarse_slots(s, sc->t1_total, sc->sort_shift + fine, slots_max);
  const unsigned long long t1_total = sc->t1_total;
  const int shift = sc->sort_shift;
  const uint32_t fmask = (1u << fine) - 1u;
  __syncthreads();
  const uint32_t slots = sh.slots;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const unsigned long long q0 = (unsigned long long)blockIdx.x * chunk;
  const unsigned long long q1 = q0 + chunk < s ? q0 + chunk : s;
  for (unsigned long long base = q0; base < q1; base += kSortTile) {
    const uint32_t n = (uint32_t)(q1 - base < (unsigned long long)kSortTile ? q1 - base : kSortTile);
    sh.cnt[tid] = 0;
    __syncthreads();
    uint32_t b[kTilePer], rank[kTilePer];
#pragma unroll
    for (int u = 0; u < kTilePer; ++u) {
      const uint32_t x = tid + u * kSortThreads;
      b[u] = 0;
      rank[u] = 0;
      if (x < n) {
        b[u] = sort_bucket(first + base + x, key, t1_total, shift);
        rank[u] = atomicAdd(&sh.cnt[b[u] >> fine], 1u);
      }
    }
    __syncthreads();
    const uint32_t mine = sh.cnt[tid];
    sh.cur[tid] = tid < nc && mine ? atomicAdd(&taken->n[tid], mine) : 0u;
    sh.off[tid] = block_exclusive_1024(mine, sh.warp_sum);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kTilePer; ++u) {
      const uint32_t x = tid + u * kSortThreads;
      if (x < n) {
        const uint32_t c = b[u] >> fine, at = sh.off[c] + rank[u];
        sh.rec[at] = ((b[u] & fmask) << kIdxBits) | (uint32_t)(base + x);
        sh.bkt[at] = (uint16_t)c;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kTilePer; ++u) {
      const uint32_t x = tid + u * kSortThreads;
      if (x < n) {
        const uint32_t c = sh.bkt[x], at = sh.cur[c] + x - sh.off[c];
        if (at < slots) rec[(size_t)c * slots + at] = sh.rec[x];
        else over[atomicAdd(&taken->over, 1u)] = make_uint2(c, sh.rec[x]);
      }
    }
    __syncthreads();
  }
}

// Step 2, coarse bucket blockIdx.x: its records by their low bits into order
// (indices alone) and the first place of each of its buckets into base
// (base[nbk] = s).  Longer than kFineStage, it is written in place order
// straight to memory.
__global__ void __launch_bounds__(kSortThreads, 2)
k_sort_fine(const DevScalars* __restrict__ sc, const uint32_t* __restrict__ rec,
            const uint2* __restrict__ over, const SortTaken* __restrict__ taken, int fine,
            unsigned long long s, unsigned long long slots_max, uint32_t* __restrict__ order,
            unsigned int* __restrict__ base) {
  extern __shared__ uint32_t stage[];
  __shared__ uint32_t cur[1 << (kSortBitsMax - kCoarseBits)];
  __shared__ uint32_t warp_sum[32], s_slots, s_p0;
  const uint32_t c = blockIdx.x, nf = 1u << fine;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  if (c + 1 == gridDim.x && tid == 0) base[(size_t)gridDim.x << fine] = (unsigned int)s;
  // The places before it: those of the coarse buckets before it.
  uint32_t before = tid < c ? taken->n[tid] : 0u;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
  if (lane == 0) warp_sum[tid >> 5] = before;
  if (tid < nf) cur[tid] = 0;
  if (tid == 0) s_slots = coarse_slots(s, sc->t1_total, sc->sort_shift + fine, slots_max);
  __syncthreads();
  if (tid < 32) {
    uint32_t v = warp_sum[tid];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (tid == 0) s_p0 = v;
  }
  const uint32_t n = taken->n[c], held = min(n, s_slots);
  const uint32_t listed = n > held ? taken->over : 0u;
  const uint32_t* __restrict__ mine = rec + (size_t)c * s_slots;
  for (uint32_t x = tid; x < held; x += kSortThreads) atomicAdd(&cur[mine[x] >> kIdxBits], 1u);
  for (uint32_t x = tid; x < listed; x += kSortThreads) {
    const uint2 e = over[x];
    if (e.x == c) atomicAdd(&cur[e.y >> kIdxBits], 1u);
  }
  __syncthreads();
  const uint32_t p0 = s_p0;
  if (tid < 32) {   // nf <= 64 counts: two per lane
    const uint32_t a = 2 * tid < nf ? cur[2 * tid] : 0u;
    const uint32_t d = 2 * tid + 1 < nf ? cur[2 * tid + 1] : 0u;
    uint32_t inc = a + d;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (tid >= o) inc += y;
    }
    const uint32_t ex = inc - a - d;
    if (2 * tid < nf) {
      cur[2 * tid] = ex;
      base[c * nf + 2 * tid] = p0 + ex;
    }
    if (2 * tid + 1 < nf) {
      cur[2 * tid + 1] = ex + a;
      base[c * nf + 2 * tid + 1] = p0 + ex + a;
    }
  }
  __syncthreads();
  uint32_t* __restrict__ out = n <= kFineStage ? stage : order + p0;
  for (uint32_t x = tid; x < held; x += kSortThreads) {
    const uint32_t r = mine[x];
    out[atomicAdd(&cur[r >> kIdxBits], 1u)] = r & kIdxMask;
  }
  for (uint32_t x = tid; x < listed; x += kSortThreads) {
    const uint2 e = over[x];
    if (e.x == c) out[atomicAdd(&cur[e.y >> kIdxBits], 1u)] = e.y & kIdxMask;
  }
  if (n > kFineStage) return;
  __syncthreads();
  for (uint32_t x = tid; x < n; x += kSortThreads) order[p0 + x] = stage[x];
}

// Diamonds in row order (dense inputs): order[q] = l - first.  Draws only:
// diamond q's hash key goes to keys[q] (EMPTY_KEY when it adds nothing:
// v = 0 or an excluded diagonal) and its increment to vals[q].  Under
// MAD_SQUARE_SYM the same increment for the pair (k, k') goes to keys[s +
// q] and vals[s + q] (Sec. 3.2.3).  k_insert adds them to X.
//
// The draws are draw_given_row's, written out for dense inputs of one type.
// Load latency binds it, with issue slots and L1 at 53 % and 63 % of their rates
// and DRAM at 17 % (560 instructions a diamond): without the branches on input
// kinds and with 32-bit totals multiplied as such (680 instructions before) the
// fused pass went from 930 to 907 us.  TB in 64-byte blocks, as the batched queries draw, is slower here
// (972 us: TB and its guides are in L2, and a block reads twice their bytes),
// and so are 7 or 8 blocks per SM (935 us).
template <typename TBV>
__global__ void __launch_bounds__(256, 6)
k_sample_sorted(const SampleParams p_, unsigned long long seed, unsigned long long first,
                unsigned long long s, const uint32_t* __restrict__ order,
                unsigned long long* __restrict__ keys, long long* __restrict__ vals) {
  const bool sqsym = (p_.flags & MAD_SQUARE_SYM) != 0;
  const SampleParams p = resolve(p_);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const int d = (int)p.d;
  bool bad = false;
  unsigned long long diag = 0;
  for (unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; q < s;
       q += stride) {
    const Uniforms u = diamond_uniforms(seed, first + __ldcs(order + q));
    Draw dr;
    {
      const int64_t i = draw_row_i(p, u.u0, &bad);
      const uint32_t* __restrict__ r2 = p.T2 + i * p.d;
      const uint32_t* __restrict__ ra = p.TA + i * p.d;
      int k, kp;
      ub2_u32(r2, ra, d, draw_target32(u.u1, __ldg(r2 + d - 1) & PREFIX_MASK),
              draw_target32(u.u3, __ldg(ra + d - 1) & PREFIX_MASK), PREFIX_MASK, &k, &kp);
      if (k >= d) { bad = true; k = d - 1; }
      if (kp >= d) { bad = true; kp = d - 1; }
      uint32_t sign = __ldg(r2 + k) ^ __ldg(ra + kp);
      const uint32_t* __restrict__ row = p.TB + (int64_t)k * p.n;
      int64_t j = ub_guided_u32(row, p.TBg + k * p.tbg_stride, (int)__ldg(p.TBg_sh + k),
                                draw_target32(u.u2, __ldg(row + p.n - 1) & PREFIX_MASK),
                                PREFIX_MASK);
      if (j >= p.n) { bad = true; j = p.n - 1; }
      sign ^= __ldg(row + j);
      const TBV b = __ldg((const TBV*)p.b_val + (int64_t)kp * p.ldb + j);
      dr.i = (uint32_t)i;
      dr.k = (uint32_t)k;
      dr.j = (uint32_t)j;
      dr.kp = (uint32_t)kp;
      dr.v = fixed_point((float)b, p.f_exp);
      if (!(p.flags & MAD_NONNEG) && (sign & SIGN_BIT)) dr.v = -dr.v;
    }
    unsigned long long key = EMPTY_KEY;
    if ((p.flags & MAD_EXCLUDE_DIAG) && dr.i == dr.j) {
      ++diag;
    } else if (dr.v != 0) {
      uint32_t a = dr.i, b = dr.j;
      if ((p.flags & MAD_GRAM) && b < a) {
        a = dr.j;
        b = dr.i;
      }
      key = ((unsigned long long)a << 32) | b;
    }
    keys[q] = key;
    vals[q] = dr.v;
    if (sqsym) {
      unsigned long long key2 = EMPTY_KEY;
      if ((p.flags & MAD_EXCLUDE_DIAG) && dr.k == dr.kp) {
        ++diag;
      } else if (dr.v != 0) {
        const uint32_t a = dr.k < dr.kp ? dr.k : dr.kp, b = dr.k < dr.kp ? dr.kp : dr.k;
        key2 = ((unsigned long long)a << 32) | b;
      }
      keys[s + q] = key2;
      vals[s + q] = dr.v;
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) diag += __shfl_xor_sync(0xFFFFFFFFu, diag, off);
  const unsigned any_bad = __ballot_sync(0xFFFFFFFFu, bad);
  if ((threadIdx.x & 31) == 0) {
    if (diag) atomicAdd(&p.sc->diag_skipped, diag);
    if (any_bad) atomicOr(&p.sc->err, DERR_SEARCH);
  }
}

// X update for the row-ordered diamonds: a lean kernel (full occupancy) so
// many inserts are in flight at once; consecutive entries share row i and
// hence its hash region.
__global__ void __launch_bounds__(256, 6)
k_insert(const SampleParams p_, const unsigned long long* __restrict__ keys,
         const long long* __restrict__ vals, unsigned long long s) {
  const SampleParams p = resolve(p_);
  Tally t;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long rounds = (s + stride - 1) / stride;
  // The next entry is loaded before the current one is inserted.
  unsigned long long key = q < s ? __ldcs(keys + q) : EMPTY_KEY;
  long long v = q < s ? __ldcs(vals + q) : 0;
  for (unsigned long long r = 0; r < rounds; ++r) {
    const unsigned long long qn = q + stride;
    const unsigned long long key_n = qn < s ? __ldcs(keys + qn) : EMPTY_KEY;
    const long long v_n = qn < s ? __ldcs(vals + qn) : 0;
    if (key != EMPTY_KEY) {
      ++t.inserted;
      const int res = hash_add(p, key, v);
      if (res == 0) t.full = true;
      if (res == 2) ++t.created;
    }
    key = key_n;
    v = v_n;
    q = qn;
  }
  flush_tally(p, t);
}

// (key, value) pairs added to X as k_insert adds drawn diamonds: partial X
// of other diamond ranges merged into this context's X (sharded runs).
// Counts the keys it creates, not diamonds.
__global__ void __launch_bounds__(256)
k_accumulate(const SampleParams p_, const unsigned long long* __restrict__ keys,
             const long long* __restrict__ vals, unsigned long long n) {
  const SampleParams p = resolve(p_);
  Tally t;
  for (unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
       q += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long key = keys[q];
    if (key == EMPTY_KEY) continue;
    const int res = hash_add(p, key, vals[q]);
    if (res == 0) t.full = true;
    if (res == 2) ++t.created;
  }
  flush_tally(p, t);
}

// ---- X from empty, one group of rows per block -----------------------------
// When a single sorted batch of diamonds fills an empty X (the fused pass),
// the home regions are written whole instead of cleared and then updated
// with global atomics.  The sort buckets are taken 2^lg_group at a time; group
// g covers the targets [g << gs, (g + 1) << gs) with gs = sort shift +
// lg_group and owns the rows whose first target lies there,
// [R[g], R[g+1]) with R[0] = 0, R[g] = 1 + #{r : T1[r] < g << gs} and
// R[last + 1] = m.  Their regions, [hreg[R[g]], hreg[R[g+1]]), are
// contiguous.  A block builds them in shared memory from the diamonds of its
// buckets (those of its last row that fall into later buckets included) and
// stores them with plain coalesced writes, so X is written once and never read
// back from DRAM.  Every key probes linearly from its home slot (home_slot) to
// the end of its group's regions; a key that finds no place before it goes to
// the overflow table after the regions, [hreg[m], hreg[m] + O), a plain
// linear-probing hash (a key in two groups or so, at the loads of 1/3 to 2/3
// that the regions are sized for).  So the regions are what k_insert would
// leave, but for those keys, and k_fold_overflow makes X a plain table again
// before anything else is added to it.  Groups whose regions exceed the
// shared-memory image are "heavy": a first kernel clears their regions and
// the diamonds of their rows are added with global atomics (the same
// probing) by whichever block holds them in its own buckets.
// Each diamond is added exactly once, so X is the same set of
// (key, sum) as the one k_insert builds (the sums are exact integers).
constexpr int kImageSlots = 3072;   // 48 KB: keys, then values
constexpr int kSpill = 32;          // slots after a group's regions in the image
constexpr int kRowCache = 256;      // owned rows whose hreg a block keeps in shared memory

// R[h] for a group boundary h (see above): 1 + #{r : T1[r] < h << gs}, read
// from the T1 guide (entry b counts the T1 entries below b << t1g_sh, and
// gs >= t1g_sh: the boundary is on a guide bucket).
__device__ __forceinline__ int64_t group_first_row(const SampleParams& p, uint32_t h,
                                                   uint32_t ngroups, int gs) {
  if (h == 0) return 0;
  if (h >= ngroups) return p.m;
  const unsigned long long t = (unsigned long long)h << gs;
  if (t > p.t1_total) return p.m;
  const int64_t r = (int64_t)__ldg(p.T1g + (t >> p.t1g_sh)) + 1;
  return r < p.m ? r : p.m;
}

// Row bounds of every group (R), its heavy flag, the sorted position where
// the diamonds it builds end (qend: its own buckets and those of its last
// row's diamonds), the clearing of heavy groups' regions and of the
// overflow table.  One warp per group.
__global__ void __launch_bounds__(256)
k_group_prep(const SampleParams p_, const unsigned int* __restrict__ base, uint32_t nbk,
             int lg_group, uint32_t ngroups, uint64_t ov_slots, int narrow,
             uint32_t* __restrict__ R, unsigned char* __restrict__ heavy,
             uint32_t* __restrict__ qend) {
  const SampleParams p = resolve(p_);
  const int lane = threadIdx.x & 31;
  const uint32_t g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int gs = p.sc->sort_shift + lg_group;
  const unsigned long long ov0 = p.hreg[p.m];
  if (ov0 + ov_slots > p.hcap_alloc) {   // (the allocation bounds the regions)
    if (g == 0 && lane == 0) atomicOr(&p.sc->err, DERR_HASH_FULL);
    return;
  }
  if (g < ngroups) {
    unsigned long long slot = 0, tend = 0;
    int64_t r = 0;
    if (lane < 2) {
      r = group_first_row(p, g + lane, ngroups, gs);
      slot = p.hreg[r];
      if (lane == 1 && r > 0) tend = p.T1[r - 1];   // where the last owned row's targets end
      if (lane == 0) R[g] = (uint32_t)r;
      if (lane == 1 && g + 1 == ngroups) R[ngroups] = (uint32_t)p.m;
    }
    const unsigned long long lo = __shfl_sync(0xFFFFFFFFu, slot, 0);
    const unsigned long long hi = __shfl_sync(0xFFFFFFFFu, slot, 1);
    const int64_t r0 = __shfl_sync(0xFFFFFFFFu, r, 0);
    const int64_t r1 = __shfl_sync(0xFFFFFFFFu, r, 1);
    // Narrow image keys name the row by its offset in the group (8 bits).
    const bool big = hi - lo > (unsigned long long)kImageSlots ||
                     (narrow && r1 - r0 >= (int64_t)kRowCache);
    if (lane == 1) {
      // The sorted position where the diamonds the group builds end: its
      // own buckets, and those of its last row.
      const int bsh = p.sc->sort_shift;
      const uint32_t b1 = (g + 1) << lg_group;
      unsigned long long be = (tend >> bsh) + ((tend & ((1ull << bsh) - 1)) ? 1 : 0);
      be = be < nbk ? be : nbk;
      qend[g] = (!big && r > r0 && be > b1) ? base[be] : base[b1];
    }
    if (lane == 0) heavy[g] = big ? 1 : 0;
    if (big)
      for (unsigned long long x = lo + lane; x < hi; x += 32) {
        p.hkeys[x] = EMPTY_KEY;
        p.hvals[x] = 0;
      }
  }
  for (unsigned long long x = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
       x < ov_slots; x += (unsigned long long)gridDim.x * blockDim.x) {
    p.hkeys[ov0 + x] = EMPTY_KEY;
    p.hvals[ov0 + x] = 0;
  }
}

// Global insert of key into [slot, hi) from slot on, then, when that is full,
// into the overflow table.  1 existing key, 2 new key, 0 both full.
__device__ __forceinline__ int add_span_or_overflow(const SampleParams& p, unsigned long long hi,
                                                    unsigned long long slot,
                                                    unsigned long long ov0, uint64_t ov_slots,
                                                    unsigned long long key, long long v) {
  if (slot < hi) {   // (hi - slot probes end before the wrap)
    const int r = hash_add_from(p.hkeys, p.hvals, slot, hi, slot, (uint32_t)(hi - slot), key, v);
    if (r) return r;
  }
  return hash_add_from(p.hkeys, p.hvals, ov0, ov0 + ov_slots, ov0 + (mix64(key) & (ov_slots - 1)),
                       (uint32_t)ov_slots, key, v);
}

// The regions of group blockIdx.x (see above).  base[b] is the first sorted
// position of bucket b (base[nbk] = the batch size); R, heavy and qend_g
// come from k_group_prep.
//
// kNarrow: the image holds 32-bit keys, (row - first owned row) << 24 | j,
// for n <= 2^24 and groups of fewer than kRowCache rows (k_group_prep makes
// larger groups heavy): the key claim is a 32-bit compare-and-swap and one
// 16-byte shared load reads four probe slots.  Otherwise the image holds
// the 64-bit keys.  The stored X holds 64-bit keys either way.
template <bool kNarrow>
__global__ void __launch_bounds__(256)
k_build_x(const SampleParams p_, const unsigned long long* __restrict__ keys,
          const long long* __restrict__ vals, const unsigned int* __restrict__ base,
          uint32_t nbk, int lg_group, uint32_t ngroups, uint64_t ov_slots,
          const uint32_t* __restrict__ R, const unsigned char* __restrict__ heavy,
          const uint32_t* __restrict__ qend_g) {
  // kImageSlots + kSpill keys (4 or 8 bytes), then as many 8-byte values.
  extern __shared__ __align__(16) unsigned long long img[];
  using IKey = typename std::conditional<kNarrow, uint32_t, unsigned long long>::type;
  constexpr IKey kEmptyI = (IKey)~(IKey)0;
  __shared__ uint32_t s_off[kRowCache + 1];   // owned rows' region offsets in the image
  const SampleParams p = resolve(p_);
  const unsigned long long ov0 = p.hreg[p.m];
  if (ov0 + ov_slots > p.hcap_alloc) return;   // reported by k_group_prep
  const uint32_t g = blockIdx.x;
  const int bsh = p.sc->sort_shift;
  const int gs = bsh + lg_group;
  const uint32_t b0 = g << lg_group;
  const uint32_t b1 = b0 + (1u << lg_group) < nbk ? b0 + (1u << lg_group) : nbk;
  // Every thread reads the group's bounds (one broadcast round trip), then
  // its regions' bounds and its first diamond.
  const uint32_t r0 = R[g], r1 = R[g + 1];
  const unsigned long long q0 = base[b0], q1 = base[b1], qend = qend_g[g];
  const bool hv = heavy[g] != 0;
  const unsigned long long lo = p.hreg[r0];
  const unsigned long long span = hv ? 0 : p.hreg[r1] - lo;
  const bool cached = r1 - r0 < (uint32_t)kRowCache;
  if (!hv && cached)
    for (uint32_t x = threadIdx.x; x <= r1 - r0; x += blockDim.x)
      s_off[x] = (uint32_t)(p.hreg[r0 + x] - lo);
  // Keys that reach the end of the regions go on into the spill slots, which
  // leave for the overflow table at the end, beside the image's stores.
  const uint32_t span32 = (uint32_t)span, end32 = hv ? 0u : span32 + kSpill;
  unsigned long long q = q0 + threadIdx.x;
  unsigned long long key = q < qend ? keys[q] : EMPTY_KEY;
  long long v = q < qend ? vals[q] : 0;
  IKey* ik = (IKey*)img;
  unsigned long long* iv = (unsigned long long*)((char*)img + (kImageSlots + kSpill) * sizeof(IKey));
  for (uint32_t x = 4 * threadIdx.x; x < end32; x += 4 * blockDim.x) {
    if (kNarrow) {
      *(uint4*)(ik + x) = make_uint4(~0u, ~0u, ~0u, ~0u);
    } else {
      *(ulonglong2*)(ik + x) = make_ulonglong2(EMPTY_KEY, EMPTY_KEY);
      *(ulonglong2*)(ik + x + 2) = make_ulonglong2(EMPTY_KEY, EMPTY_KEY);
    }
    *(ulonglong2*)(iv + x) = make_ulonglong2(0, 0);
    *(ulonglong2*)(iv + x + 2) = make_ulonglong2(0, 0);
  }
  __syncthreads();
  Tally t;
  for (; q < qend; q += blockDim.x) {
    // The next diamond is loaded before this one is added.
    const unsigned long long qn = q + blockDim.x;
    const unsigned long long key_n = qn < qend ? keys[qn] : EMPTY_KEY;
    const long long v_n = qn < qend ? vals[qn] : 0;
    const unsigned long long k = key;
    const long long w = v;
    key = key_n;
    v = v_n;
    if (k == EMPTY_KEY) continue;
    const uint32_t i = (uint32_t)(k >> 32);
    const bool own = !hv && i >= r0 && i < r1;
    int res;
    if (own) {
      // Linear probe of the image from the home slot to its end, four slots
      // per step (two 16-byte shared loads; regions start on 4-slot groups).
      // The probes left end the loop at the image's end, so the wraps below are
      // never taken; the loop compiled without them costs the pass 3 us, and
      // ended by the position instead of the count 15 us (849 -> 852, 865).
      // A stale EMPTY is caught by the CAS; a key once set never changes.
      // Image positions are 32-bit (the image holds kImageSlots slots).
      uint32_t roff, rsz;
      if (cached) {
        roff = s_off[i - r0];
        rsz = s_off[i - r0 + 1] - roff;
      } else {
        const unsigned long long a = __ldg(p.hreg + i);
        roff = (uint32_t)(a - lo);
        rsz = (uint32_t)(__ldg(p.hreg + i + 1) - a);
      }
      uint32_t x = roff + (uint32_t)region_offset((uint32_t)k, rsz);
      const IKey kk = kNarrow ? (IKey)(((i - r0) << 24) | (uint32_t)k) : (IKey)k;
      res = 0;
      for (uint32_t probes = 0, left = end32 - x; probes < left;) {
        const uint32_t gx = x & ~3u;
        IKey k4[4];
        if (kNarrow) {
          const uint4 ka = *(const uint4*)(ik + gx);
          k4[0] = (IKey)ka.x; k4[1] = (IKey)ka.y; k4[2] = (IKey)ka.z; k4[3] = (IKey)ka.w;
        } else {
          const ulonglong2 ka = *(const ulonglong2*)(ik + gx);
          const ulonglong2 kb = *(const ulonglong2*)(ik + gx + 2);
          k4[0] = (IKey)ka.x; k4[1] = (IKey)ka.y; k4[2] = (IKey)kb.x; k4[3] = (IKey)kb.y;
        }
        const uint32_t start = x - gx;
        uint32_t pick = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u)
          pick = ((uint32_t)u >= start && (k4[u] == kk || k4[u] == kEmptyI)) ? (uint32_t)u : pick;
        if (pick == 4) {
          probes += 4 - start;
          x = gx + 4 < end32 ? gx + 4 : 0;
          continue;
        }
        probes += pick - start + 1;
        IKey cur = k4[0];
#pragma unroll
        for (int u = 1; u < 4; ++u) cur = (uint32_t)u == pick ? k4[u] : cur;
        const uint32_t slot = gx + pick;
        const IKey prev = cur == kk ? kk : atomicCAS(ik + slot, kEmptyI, kk);
        if (prev == kEmptyI || prev == kk) {
          // The 64-bit sum as two 32-bit shared atomics: the low word's own
          // carry goes into the high word, so the total is the exact sum.
          unsigned int* h2 = (unsigned int*)(iv + slot);
          const unsigned int wlo = (unsigned int)w;
          const unsigned int whi = (unsigned int)((unsigned long long)w >> 32);
          const unsigned int olo = atomicAdd(h2, wlo);
          atomicAdd(h2 + 1, whi + (olo + wlo < olo ? 1u : 0u));
          res = prev == kEmptyI ? 2 : 1;
          break;
        }
        x = slot + 1 < end32 ? slot + 1 : 0;   // taken by another key: go on after it
      }
      if (res == 0) res = add_span_or_overflow(p, 0, 0, ov0, ov_slots, k, w);
    } else {
      if (q >= q1) continue;   // the owner's extension: not this block's
      const unsigned long long ex = i ? __ldg(p.T1 + i - 1) : 0ull;
      unsigned long long og = ex >> gs;
      og = og < ngroups - 1 ? og : ngroups - 1;
      if (!heavy[og]) continue;   // its owner builds it
      const unsigned long long rlo = __ldg(p.hreg + i), rhi = __ldg(p.hreg + i + 1);
      const unsigned long long home = rlo + region_offset((uint32_t)k, rhi - rlo);
      res = add_span_or_overflow(p, p.hreg[R[og + 1]], home, ov0, ov_slots, k, w);
    }
    ++t.inserted;
    if (res == 0) t.full = true;
    if (res == 2) ++t.created;
  }
  __syncthreads();
  // Image keys widened back to (i << 32) | j.
  auto wide = [&](uint32_t x) -> unsigned long long {
    const IKey a = ik[x];
    if (a == kEmptyI) return EMPTY_KEY;
    return kNarrow ? ((unsigned long long)(r0 + ((uint32_t)a >> 24)) << 32) | ((uint32_t)a & 0xFFFFFFu)
                   : (unsigned long long)a;
  };
  // A spilled key is in no other block's hands: a claimed slot of the overflow
  // table is its own, and the claim's round trip passes beside the stores below.
  unsigned long long spilled = EMPTY_KEY, at = 0, prev = EMPTY_KEY;
  if (threadIdx.x < kSpill && !hv) spilled = wide(span32 + threadIdx.x);
  if (spilled != EMPTY_KEY) {
    at = mix64(spilled) & (ov_slots - 1);
    prev = atomicCAS(p.hkeys + ov0 + at, EMPTY_KEY, spilled);
  }
  // The image, 16 bytes per store (regions start on 4-slot groups).
  for (uint32_t x = 2 * threadIdx.x; x < span32; x += 2 * blockDim.x) {
    *(ulonglong2*)(p.hkeys + lo + x) = make_ulonglong2(wide(x), wide(x + 1));
    *(longlong2*)(p.hvals + lo + x) = make_longlong2((long long)iv[x], (long long)iv[x + 1]);
  }
  if (spilled != EMPTY_KEY) {
    for (uint64_t probes = 1; prev != EMPTY_KEY && probes < ov_slots; ++probes) {
      at = (at + 1) & (ov_slots - 1);
      prev = atomicCAS(p.hkeys + ov0 + at, EMPTY_KEY, spilled);
    }
    if (prev == EMPTY_KEY) p.hvals[ov0 + at] = (long long)iv[span32 + threadIdx.x];
    else t.full = true;
  }
  flush_tally_block(p, t);
}

// The overflow table's keys moved into the regions, where k_insert and
// k_accumulate look for them: X is a plain table afterwards.  (Each key is in
// one place, so none is counted as new; one that finds no place stays and is
// reported.)
__global__ void __launch_bounds__(256)
k_fold_overflow(const SampleParams p_, uint64_t ov_slots) {
  const SampleParams p = resolve(p_);
  const unsigned long long ov0 = p.hreg[p.m];
  if (ov0 + ov_slots > p.hcap_alloc) return;   // reported by k_group_prep
  for (unsigned long long x = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
       x < ov_slots; x += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long key = p.hkeys[ov0 + x];
    if (key == EMPTY_KEY) continue;
    if (hash_add(p, key, p.hvals[ov0 + x]) == 0) {
      atomicOr(&p.sc->err, DERR_HASH_FULL);
      continue;
    }
    p.hkeys[ov0 + x] = EMPTY_KEY;
    p.hvals[ov0 + x] = 0;
  }
}

// Diagnostic twin of k_sample: writes each diamond's draws instead of
// accumulating them.
__global__ void __launch_bounds__(256)
k_draws(const SampleParams p_, unsigned long long seed, unsigned long long first,
        const unsigned long long* __restrict__ ells, unsigned long long count, uint32_t* oi,
        uint32_t* ok, uint32_t* oj, uint32_t* okp, long long* ov) {
  const SampleParams p = resolve(p_);
  bool bad = false;
  for (unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; q < count;
       q += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long ell = ells ? ells[q] : first + q;
    const Draw dr = draw_one(p, seed, ell, &bad);
    oi[q] = dr.i;
    ok[q] = dr.k;
    oj[q] = dr.j;
    okp[q] = dr.kp;
    ov[q] = dr.v;
  }
  if (bad) atomicOr(&p.sc->err, DERR_SEARCH);
}

// Resident 256-thread blocks of `kernel` on the whole GPU (queried once
// per kernel; one process drives one device).
template <auto kernel>
int full_grid() {
  static int cached = 0;
  if (cached) return cached;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  cached = sms * per_sm;
  return cached;
}

unsigned grid_of(unsigned long long work, int full) {
  const unsigned long long need = (work + 255) / 256;
  return (unsigned)(need < (unsigned long long)full ? (need ? need : 1) : full);
}

// Diamonds per sorted batch (bounds the scratch at 20 bytes per diamond).
constexpr unsigned long long kSortBatch = 1ull << 26;

// Pilot for hash sizing: counts the diamonds that would be inserted.
template <bool kRows>
__global__ void __launch_bounds__(256)
k_pilot(const SampleParams p_, unsigned long long seed, unsigned long long n,
        unsigned long long* __restrict__ hits) {
  const SampleParams p = resolve(p_);
  bool bad = false;
  unsigned long long c = 0;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long rounds = (n + stride - 1) / stride;
  unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (unsigned long long r = 0; r < rounds; ++r, q += stride) {
    const bool valid = q < n;
    Draw dr{};
    if (kRows) dr = draw_rows<false>(p, valid, seed, q, &bad);
    else if (valid) dr = draw_one_as<false>(p, seed, q, &bad);
    if (!valid) dr.v = 0;
    c += (dr.v != 0 && !((p.flags & MAD_EXCLUDE_DIAG) && dr.i == dr.j)) ? 1 : 0;
    if (p.flags & MAD_SQUARE_SYM)
      c += (dr.v != 0 && !((p.flags & MAD_EXCLUDE_DIAG) && dr.k == dr.kp)) ? 1 : 0;
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(hits, c);
  if (bad) atomicOr(&p.sc->err, DERR_SEARCH);
}

// Caller's profiling event q (if set) on the sampling stream.
void phase_event(const mad_ctx* ctx, uint32_t q, cudaStream_t st) {
  if (q < ctx->n_phase_ev && ctx->phase_ev[q]) cudaEventRecord(ctx->phase_ev[q], st);
}

}  // namespace

SampleParams make_params(const mad_ctx* ctx) {
  SampleParams p;
  p.a_val = ctx->A.values;
  p.a_ptr = ctx->A.rowptr;
  p.a_col = ctx->A.colidx;
  p.m = ctx->m;
  p.d = ctx->d;
  p.lda = ctx->A.ld;
  p.b_val = ctx->B.values;
  p.b_ptr = ctx->B.rowptr;
  p.b_col = ctx->B.colidx;
  p.n = ctx->n;
  p.ldb = ctx->B.ld;
  p.T1 = ctx->T1;
  p.T2 = ctx->T2;
  p.TA = ctx->TA;
  p.TB = ctx->TB;
  p.t1_total = ctx->t1_total;
  p.T1g = ctx->T1g;
  p.t1g_sh = ctx->t1g_sh;
  p.T2g_ptr = ctx->T2g_ptr;
  p.T2g = ctx->T2g;
  p.T2g_sh = ctx->T2g_sh;
  p.rdesc = ctx->rdesc;
  p.brow = ctx->brow;
  p.bloom = ctx->bloom;
  p.bloom_shift = 40 - ctx->bloom_lg;
  p.TBg = ctx->TBg;
  p.tbg_stride = ctx->tbg_stride;
  p.TBg_sh = ctx->TBg_sh;
  p.tb_blocks = ctx->tb_blocks;
  p.tb_row = ctx->tb_row;
  p.f_exp = ctx->f;
  p.hkeys = ctx->hkeys;
  p.hvals = ctx->hvals;
  p.hreg = ctx->hreg;
  p.hmask = ctx->hcap - 1;
  p.hcap = ctx->hcap;
  p.hcap_alloc = ctx->hcap_alloc;
  p.max_probe = (uint32_t)(ctx->hcap < 4096 ? ctx->hcap : 4096);
  p.regioned = ctx->regioned ? 1 : 0;
  p.dense = ctx->dense ? 1 : 0;
  p.a_f64 = ctx->A.dt == MAD_F64;
  p.b_f64 = ctx->B.dt == MAD_F64;
  p.integer = ctx->integer ? 1 : 0;
  p.flags = ctx->flags;
  p.sc = ctx->sc;
  p.alias = (ctx->flags & MAD_ALIAS) && ctx->al[kAlT1] ? 1 : 0;
  for (int f = 0; f < 4; ++f) {
    p.al[f] = ctx->al[f];
    p.al_seg[f] = ctx->al_seg[f];
    p.al_row[f] = ctx->al_row[f];
    p.al_nseg[f] = ctx->al_nseg[f];
  }
  return p;
}

mad_status pilot_inserts(mad_ctx* ctx, uint64_t n, uint64_t* hits, cudaStream_t st) {
  mad_status rs = ensure_scratch(ctx, 256, st);
  if (rs != MAD_OK) return rs;
  unsigned long long* dev = (unsigned long long*)ctx->scratch;
  cudaMemsetAsync(dev, 0, sizeof(unsigned long long), st);
  const SampleParams p = make_params(ctx);
  if (p.rdesc)
    k_pilot<true><<<grid_of(n, full_grid<k_pilot<true>>()), 256, 0, st>>>(
        p, 0x9E3779B97F4A7C15ull, n, dev);
  else
    k_pilot<false><<<grid_of(n, full_grid<k_pilot<false>>()), 256, 0, st>>>(
        p, 0x9E3779B97F4A7C15ull, n, dev);
  count_launch(ctx);
  unsigned long long h = 0;
  cudaMemcpyAsync(&h, dev, sizeof(h), cudaMemcpyDeviceToHost, st);
  const cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e);
  *hits = h;
  return MAD_OK;
}

int sort_bits(int64_t m) {
  int lg = 0;
  while (lg < kSortBitsMax && (1ll << lg) < m) ++lg;
  return lg;
}

uint64_t sort_buckets(int64_t m) { return 1ull << sort_bits(m); }

// Blocks of the sort (two per SM).
int sort_blocks() {
  static int blocks = 0;
  if (!blocks) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    blocks = 2 * (sms < 1 ? 1 : sms);
  }
  return blocks;
}

// Slots of the coarse buckets together (coarse_slots): the diamonds, one more
// bucket of at most 2 s / nc, and three deviations for each.
uint64_t sort_slots(uint64_t nbk, uint64_t batch) {
  const uint64_t nc = std::min<uint64_t>(nbk, 1ull << kCoarseBits);
  const double most = 2.0 * (double)batch / (double)nc;
  return batch + (uint64_t)most + nc * ((uint64_t)(3.0 * std::sqrt(most)) + 2);
}

// Scratch of the sort and the draws for one batch: the coarse buckets' counts,
// the bucket offsets, the records in coarse order, the diamond indices in bucket
// order, and each diamond's key and increment (the sort's list of records beyond
// their slots uses the keys' memory before them).
struct SortScratch {
  SortTaken* taken;
  unsigned int* base;
  uint32_t* rec;
  uint32_t* order;
  unsigned long long* keys;
  long long* vals;
  uint32_t* R;              // row bounds of the X builder's groups
  unsigned char* heavy;     // their heavy flags
  uint32_t* qend;           // where the diamonds each group builds end
  size_t bytes;
};

// recs: records per diamond (2 under MAD_SQUARE_SYM).
SortScratch carve_sort(void* p, uint64_t nbk, uint64_t batch, int recs) {
  SortScratch c;
  char* b = (char*)p;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = b ? b + off : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return (void*)q;
  };
  c.taken = (SortTaken*)take(sizeof(SortTaken));
  c.base = (unsigned int*)take((nbk + 1) * sizeof(unsigned int));
  c.rec = (uint32_t*)take(sort_slots(nbk, batch) * sizeof(uint32_t));
  c.order = (uint32_t*)take(batch * sizeof(uint32_t));
  c.keys = (unsigned long long*)take(batch * recs * sizeof(unsigned long long));
  c.vals = (long long*)take(batch * recs * sizeof(long long));
  c.R = (uint32_t*)take((nbk + 1) * sizeof(uint32_t));
  c.heavy = (unsigned char*)take(nbk);
  c.qend = (uint32_t*)take(nbk * sizeof(uint32_t));
  c.bytes = off;
  return c;
}

int sort_records(const mad_ctx* ctx) { return (ctx->flags & MAD_SQUARE_SYM) ? 2 : 1; }

size_t sample_scratch_bytes(const mad_ctx* ctx, uint64_t s) {
  if (!ctx->dense || s == 0) return 0;
  const uint64_t batch = s < kSortBatch ? s : kSortBatch;
  return carve_sort(nullptr, sort_buckets(ctx->m), batch, sort_records(ctx)).bytes;
}

// Buckets per group of the X builder: about 640 diamonds of s_max per group
// (regions of about 1300 slots against the 3072-slot image).
int build_group_log2(uint64_t nbk, uint64_t s_max) {
  int lg = 0;
  while ((2ull << lg) <= nbk && (2ull << lg) * s_max <= 640ull * nbk) ++lg;
  return lg;
}

bool x_builder_applies(const mad_ctx* ctx, uint64_t s) {
  return ctx->dense && ctx->regioned && ctx->hov > 0 && s > 0 && s <= kSortBatch &&
         !(ctx->flags & MAD_GRAM);
}

mad_status sample_impl(mad_ctx* ctx, uint64_t s, uint64_t seed, uint64_t first, cudaStream_t st,
                       bool fresh_x) {
  if (s == 0) return MAD_OK;
  if (ctx->flags & MAD_WEDGE) return wedge_sample_impl(ctx, s, seed, first, st);
  const SampleParams p = make_params(ctx);
  // 0/1 inputs, and alias draws (their row is not monotone in the uniform,
  // so the row-order sort does not apply): diamonds in index order.
  if (!ctx->dense || p.alias) {
    phase_event(ctx, 0, st);
    phase_event(ctx, 1, st);
    if (p.rdesc) {
      // The filter's words are read evenly, the rows' tables by the rows' weights:
      // where they do not fit into L2 together, the words do not stay there (1e8
      // diamonds, 160 + 64 MB of tables and words: 4.68 -> 4.44 ms; 2e7 on 32 + 16
      // MB, which fit: 0.838 -> 0.849 with the same hint).
      int dev = 0, l2 = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
      const uint64_t bytes =
          4 * (uint64_t)(ctx->nnz_a + ctx->nnz_b) + (p.bloom ? 8ull << ctx->bloom_lg : 0ull);
      if (p.bloom && bytes > (uint64_t)l2)
        k_sample_rows<true><<<grid_of(s, full_grid<k_sample_rows<true>>()), 256, 0, st>>>(
            p, seed, first, s);
      else
        k_sample_rows<false><<<grid_of(s, full_grid<k_sample_rows<false>>()), 256, 0, st>>>(
            p, seed, first, s);
    } else if (p.alias)
      k_sample<true><<<grid_of(s, full_grid<k_sample<true>>()), 256, 0, st>>>(p, seed, first, s);
    else
      k_sample<false><<<grid_of(s, full_grid<k_sample<false>>()), 256, 0, st>>>(p, seed, first, s);
    count_launch(ctx);
    phase_event(ctx, 2, st);
    phase_event(ctx, 3, st);
    return cuda_status(cudaGetLastError());
  }
  const int full_insert = full_grid<k_insert>();
  const uint64_t nbk = sort_buckets(ctx->m);
  const int blocks = sort_blocks();
  const int bits = sort_bits(ctx->m);
  const int coarse = bits < kCoarseBits ? bits : kCoarseBits, fine = bits - coarse;
  if (!ctx->sort_smem) {
    cudaFuncSetAttribute(k_sort_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(SortTile));
    cudaFuncSetAttribute(k_sort_fine, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kFineStage * sizeof(uint32_t)));
    ctx->sort_smem = true;
  }
  const uint64_t batch = s < kSortBatch ? s : kSortBatch;
  // An empty X filled by one batch, keys owned by their drawn row: the
  // regions are built whole (k_build_x); otherwise k_insert adds to X.
  const bool build_x = fresh_x && x_builder_applies(ctx, s);
  // Narrow image keys when every column index fits in 24 bits.
  const bool narrow = ctx->n <= (1ll << 24);
  const size_t image_smem =
      (size_t)(kImageSlots + kSpill) * ((narrow ? sizeof(uint32_t) : sizeof(unsigned long long)) +
                             sizeof(unsigned long long));
  if (build_x && !ctx->image_smem) {
    const int wide_smem = (int)(2 * (size_t)(kImageSlots + kSpill) * sizeof(unsigned long long));
    cudaFuncSetAttribute(k_build_x<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem);
    cudaFuncSetAttribute(k_build_x<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem);
    ctx->image_smem = true;
  }
  mad_status rs = ensure_scratch(ctx, sample_scratch_bytes(ctx, s), st);
  if (rs != MAD_OK) return rs;
  const SortScratch w = carve_sort(ctx->scratch, nbk, batch, sort_records(ctx));
  for (uint64_t done = 0; done < s; done += batch) {
    const uint64_t n = (s - done) < batch ? (s - done) : batch;
    phase_event(ctx, 0, st);
    const unsigned long long chunk = (n + blocks - 1) / blocks;
    const uint64_t slots = sort_slots(nbk, batch);
    cudaMemsetAsync(w.taken, 0, sizeof(SortTaken), st);
    k_sort_scatter<<<blocks, kSortThreads, sizeof(SortTile), st>>>(
        ctx->sc, seed, first + done, n, chunk, coarse, fine, slots, w.taken, w.rec,
        (uint2*)w.keys);
    k_sort_fine<<<1u << coarse, kSortThreads, kFineStage * sizeof(uint32_t), st>>>(
        ctx->sc, w.rec, (const uint2*)w.keys, w.taken, fine, n, slots, w.order, w.base);
    count_launch(ctx, 2);
    phase_event(ctx, 1, st);
    if (ctx->B.dt == MAD_F64)
      k_sample_sorted<double><<<grid_of(n, full_grid<k_sample_sorted<double>>()), 256, 0, st>>>(
          p, seed, first + done, n, w.order, w.keys, w.vals);
    else
      k_sample_sorted<float><<<grid_of(n, full_grid<k_sample_sorted<float>>()), 256, 0, st>>>(
          p, seed, first + done, n, w.order, w.keys, w.vals);
    count_launch(ctx);
    phase_event(ctx, 2, st);
    if (build_x) {
      const int lg = build_group_log2(nbk, ctx->s_max);
      const uint32_t ngroups = (uint32_t)(nbk >> lg);
      k_group_prep<<<(ngroups + 7) / 8, 256, 0, st>>>(p, w.base, (uint32_t)nbk, lg, ngroups,
                                                      ctx->hov, narrow ? 1 : 0, w.R, w.heavy,
                                                      w.qend);
      if (narrow)
        k_build_x<true><<<ngroups, 256, image_smem, st>>>(p, w.keys, w.vals, w.base,
                                                          (uint32_t)nbk, lg, ngroups, ctx->hov,
                                                          w.R, w.heavy, w.qend);
      else
        k_build_x<false><<<ngroups, 256, image_smem, st>>>(p, w.keys, w.vals, w.base,
                                                           (uint32_t)nbk, lg, ngroups, ctx->hov,
                                                           w.R, w.heavy, w.qend);
      count_launch(ctx, 2);
    } else {
      k_insert<<<grid_of(n, full_insert), 256, 0, st>>>(p, w.keys, w.vals,
                                                        n * (uint64_t)sort_records(ctx));
      count_launch(ctx);
    }
    phase_event(ctx, 3, st);
  }
  return cuda_status(cudaGetLastError());
}

mad_status fold_overflow(mad_ctx* ctx, cudaStream_t st) {
  if (!x_builder_applies(ctx, ctx->s_max)) return MAD_OK;   // X is never built whole
  k_fold_overflow<<<grid_of(ctx->hov, full_grid<k_fold_overflow>()), 256, 0, st>>>(
      make_params(ctx), ctx->hov);
  count_launch(ctx);
  return cuda_status(cudaGetLastError());
}

mad_status accumulate_pairs(mad_ctx* ctx, const uint64_t* keys, const int64_t* vals, uint64_t n,
                            cudaStream_t st) {
  if (n == 0) return MAD_OK;
  const SampleParams p = make_params(ctx);
  k_accumulate<<<grid_of(n, full_grid<k_accumulate>()), 256, 0, st>>>(
      p, (const unsigned long long*)keys, (const long long*)vals, n);
  count_launch(ctx);
  return cuda_status(cudaGetLastError());
}

mad_status debug_draws_impl(mad_ctx* ctx, uint64_t seed, uint64_t first, const uint64_t* ells,
                            uint64_t count, uint32_t* oi, uint32_t* ok, uint32_t* oj,
                            uint32_t* okp, int64_t* ov, cudaStream_t st) {
  if (count == 0) return MAD_OK;
  if (ctx->flags & MAD_WEDGE)
    return wedge_draws_impl(ctx, seed, first, ells, count, oi, ok, oj, okp, ov, st);
  const SampleParams p = make_params(ctx);
  const unsigned long long blocks = (count + 255) / 256;
  k_draws<<<(unsigned)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, st>>>(
      p, seed, first, (const unsigned long long*)ells, count, oi, ok, oj, okp, (long long*)ov);
  count_launch(ctx);
  return cuda_status(cudaGetLastError());
}

}  // namespace mad
