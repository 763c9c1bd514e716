// Batched queries: many instances A = Q[q] (1 x d) against one item matrix B
// (d x n), each a complete run of Alg. 2 and Alg. 3 with its own budget.
//
// With m = 1 the stage-1 draw of the center edge always returns the query's
// row, so diamond l of query q needs only the uniforms of k, j and k' (the
// Philox stream of seed + q, counter l, exactly as a single-query run) and
// the rest of the loop body is the dense path's: k from the query's T2 row,
// j from row k of TB (a guided search: n is large), k' from its TA row, the
// increment from B.
//
// A batch is three kernels, and X never exists as a whole.
//  1. k_mips_draw: a block takes a chunk of one query's diamonds, with the
//     query's T2 and TA rows in shared memory, and leaves a record (j, signed
//     b_k'j) per diamond, grouped by part: the j of a query are split by a hash
//     into parts of at most about kPartKeys distinct columns.
//  2. k_mips_parts: a block per (query, part) gathers the part's records from
//     the query's chunks, sums them per column in a shared-memory table
//     (exact 64-bit sums) and keeps the columns that can be among the
//     query's t' largest positive x.
//  3. k_mips_final: a block per query merges its parts' lists into the t'
//     largest x by (x desc, j asc), rescores them exactly and keeps the t
//     largest |c|.
// Against one hash region of 2 to 4 s_q slots of 16 bytes per query in
// global memory (cleared, filled with global atomics and read back three times
// by one block per query), a diamond moves 16 bytes of records in and out
// instead of about 250, no global atomic is left, and a query's selection is
// spread over its parts.  Measured on one GB300: 1e4 queries of 5e4 diamonds
// on 1e6 items x 300, 142 -> 32.3 ms; 61 queries on 50,021 x 100, 1300 -> 200 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "draw.cuh"
#include "mad_device.cuh"
#include "mad_internal.cuh"
#include "mips_shape.h"

namespace mad {

// One query of a planned batch: budget, first record, first entry of its
// chunks' part offsets, first candidate; parts, first part (over the batch),
// first chunk, candidates a part may keep.
struct MipsQuery {
  unsigned long long s, rec, off, cand;
  uint32_t parts, ubase, cbase, cap;
};

namespace {

constexpr int kPartThreads = 512;
constexpr int kGroup = kPartThreads;         // chunks of a part scanned together
constexpr int kAhead = 4;                    // records of a thread in flight
constexpr int kSlots = 8192;                 // largest table of a part (96 KB: two blocks per SM)
constexpr int kTPrimeMax = 1024;             // largest t' of a batch
constexpr int kSlack = 32;                   // columns a part may keep beyond t'
constexpr int kBins = 2048;                  // digits of the threshold search (11 bits)
constexpr int kSortMax = 2048;               // >= kTPrimeMax + kSlack
constexpr uint32_t kNoKey = 0xFFFFFFFFu;     // (columns are below 2^31)
static_assert(4 * kPartThreads <= kBins, "the warps' queues (64 records each) share the histogram's words");

// Upper bounds in two shared-memory rows of the same length (independent
// chains), as ub2_u32.
__device__ __forceinline__ void ub2_shared(const uint32_t* P, const uint32_t* Q, int len,
                                           uint32_t tp, uint32_t tq, int* op, int* oq) {
  int a = 0, b = 0;
  for (int step = 1 << (31 - __clz(len)); step > 0; step >>= 1) {
    const int na = a + step, nb = b + step;
    const uint32_t va = P[(na <= len ? na : len) - 1] & PREFIX_MASK;
    const uint32_t vb = Q[(nb <= len ? nb : len) - 1] & PREFIX_MASK;
    a = (na <= len && va <= tp) ? na : a;
    b = (nb <= len && vb <= tq) ? nb : b;
  }
  *op = a;
  *oq = b;
}

// The j search where the blocks are not built (tb_blocks_apply): row k's guide,
// and its window of TB 16 bytes at a time: at most kQuads aligned quads hold a
// window of 17 or fewer entries.  Entries of the row before the window are at
// most the target and entries after it above, so whole quads are counted and
// only the row's own ends are checked (TB is allocated with four entries of
// padding).
constexpr int kQuads = 5;
__device__ __forceinline__ int64_t ub_tb(const SampleParams& p, int64_t k, uint32_t target) {
  const uint32_t* __restrict__ G = p.TBg + k * p.tbg_stride;
  const uint32_t b = target >> (int)__ldg(p.TBg_sh + k);
  const uint32_t lo = __ldg(G + b), hi = __ldg(G + b + 1);
  const int64_t row = k * p.n;
  if (hi - lo > 17u)
    return (int64_t)lo + ub_u32(p.TB + row + lo, (int)(hi - lo), target, PREFIX_MASK);
  const int64_t e0 = (row + lo) & ~(int64_t)3;
  const int quads = (int)((row + hi - e0 + 3) >> 2);
  uint4 w[kQuads];
#pragma unroll
  for (int q = 0; q < kQuads; ++q)
    if (q < quads) w[q] = __ldg(reinterpret_cast<const uint4*>(p.TB + e0) + q);
  const int64_t first = e0 - row;   // (below 0 by up to 3 in a row's first quad)
  int cnt = 0;
  const bool inner = first >= 0 && first + 4 * kQuads <= p.n;
#pragma unroll
  for (int q = 0; q < kQuads; ++q) {
    if (q < quads) {
      const uint32_t v[4] = {w[q].x, w[q].y, w[q].z, w[q].w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int64_t at = first + 4 * q + c;
        const bool in_row = inner || (at >= 0 && at < p.n);
        cnt += (in_row && (v[c] & PREFIX_MASK) <= target) ? 1 : 0;
      }
    }
  }
  return (first > 0 ? first : 0) + cnt;
}

// The part of column j among `parts`: the high bits of a mix of j (the
// tables use its low bits).
__device__ __forceinline__ uint32_t part_of(uint32_t h, uint32_t parts) {
  return __umulhi(h, parts);
}

// Step 1 (see above).  chunk c: diamonds (c - cbase) * chunk ... of query
// chunk_q[c].  Shared memory: the query's T2 and TA rows, the chunk's records,
// their parts and ranks, the parts' counts.  Bound by DRAM's random reads: per
// diamond a block of TB (64 bytes) and b_k'j (a sector, fetched as 64 bytes) for
// a million items, 4.5e10 of them a second (random reads reach 3.9e10 over 4.4 GB
// and more where items repeat); 2 to 5 resident blocks per SM measure
// the same, 6 leave too little L1 (8.46 instead of 6.59 ms for 1500 queries).
template <bool kBlocks>
__global__ void __launch_bounds__(kDrawThreads, 4)
k_mips_draw(const SampleParams p, unsigned long long seed, const MipsQuery* __restrict__ queries,
            const uint32_t* __restrict__ chunk_q, unsigned long long nchunks, int mult,
            uint32_t max_parts, uint2* __restrict__ rec, uint16_t* __restrict__ off) {
  extern __shared__ __align__(16) unsigned char draw_smem[];
  const int chunk = mult * kDrawThreads;
  const int d = (int)p.d;
  uint2* srec = (uint2*)draw_smem;                    // chunk records
  uint2* stb = srec + chunk;                          // total and mul of TB's rows
  uint32_t* splace = (uint32_t*)(stb + d);            // part << 16 | rank in it
  uint32_t* scnt = splace + chunk;                    // max_parts counts, then offsets
  uint32_t* s2 = scnt + max_parts + 1;                // T2 row
  uint32_t* sa = s2 + d;                              // TA row
  uint16_t* sord = (uint16_t*)(sa + d);               // source of each place
  __shared__ uint32_t warp_sum[kDrawThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t nb = tb_blocks(p.n);
  bool bad = false;
  if (kBlocks)
    for (int x = tid; x < d; x += kDrawThreads) stb[x] = __ldg(p.tb_row + x);
  for (unsigned long long c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const uint32_t q = __ldg(chunk_q + c);
    const MipsQuery mq = queries[q];
    const unsigned long long l0 = (c - mq.cbase) * (unsigned long long)chunk;
    const int cnt = (int)(mq.s - l0 < (unsigned long long)chunk ? mq.s - l0
                                                                 : (unsigned long long)chunk);
    for (int x = tid; x < d; x += kDrawThreads) {
      s2[x] = __ldg(p.T2 + (int64_t)q * d + x);
      sa[x] = __ldg(p.TA + (int64_t)q * d + x);
    }
    for (uint32_t x = tid; x < mq.parts; x += kDrawThreads) scnt[x] = 0;
    __syncthreads();
    const uint32_t t2tot = s2[d - 1] & PREFIX_MASK, tatot = sa[d - 1] & PREFIX_MASK;
    // (Whole warps: the blocks of TB are read by a warp's lanes together.)
    for (int x0 = warp * 32; x0 < cnt; x0 += kDrawThreads) {
      const int x = x0 + lane;
      const Uniforms un = diamond_uniforms(seed + q, l0 + (x < cnt ? x : cnt - 1));
      int k, kp;
      ub2_shared(s2, sa, d, draw_target32(un.u1, t2tot),
                 draw_target32(un.u3, tatot), &k, &kp);
      if (k >= d) { bad = true; k = d - 1; }
      if (kp >= d) { bad = true; kp = d - 1; }
      uint32_t sj;
      int64_t j;
      if (kBlocks) {
        const uint2 tb = stb[k];
        j = ub_block(p, nb, k, tb.y, draw_target32(un.u2, tb.x), &sj);
        if (j >= p.n) { bad = true; j = p.n - 1; }
      } else {
        const int64_t row = (int64_t)k * p.n;
        const uint32_t tot = __ldg(p.TB + row + p.n - 1) & PREFIX_MASK;
        j = ub_tb(p, k, draw_target32(un.u2, tot));
        if (j >= p.n) { bad = true; j = p.n - 1; }
        sj = __ldg(p.TB + row + j) & SIGN_BIT;
      }
      const uint32_t sign = sj ^ ((s2[k] ^ sa[kp]) & SIGN_BIT);
      const float b = __ldg((const float*)p.b_val + (int64_t)kp * p.ldb + j);
      if (x >= cnt) continue;
      const uint32_t part = part_of(fmix32((uint32_t)j), mq.parts);
      const uint32_t rank = atomicAdd(&scnt[part], 1u);
      srec[x] = make_uint2((uint32_t)j, __float_as_uint(b) ^ sign);
      splace[x] = (part << 16) | rank;
    }
    __syncthreads();
    // Exclusive scan of the counts (each thread a run of parts).
    const uint32_t per = (mq.parts + kDrawThreads - 1) / kDrawThreads;
    uint32_t mine = 0;
    for (uint32_t x = tid * per; x < min((tid + 1) * per, mq.parts); ++x) mine += scnt[x];
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    uint32_t run = inc - mine;
    for (int w = 0; w < warp; ++w) run += warp_sum[w];
    uint16_t* __restrict__ o = off + mq.off + (c - mq.cbase) * (unsigned long long)(mq.parts + 1);
    for (uint32_t x = tid * per; x < min((tid + 1) * per, mq.parts); ++x) {
      const uint32_t v = scnt[x];
      scnt[x] = run;
      o[x] = (uint16_t)run;
      run += v;
    }
    if (tid == 0) o[mq.parts] = (uint16_t)cnt;
    __syncthreads();
    for (int x = tid; x < cnt; x += kDrawThreads) {
      const uint32_t pl = splace[x];
      sord[scnt[pl >> 16] + (pl & 0xFFFFu)] = (uint16_t)x;
    }
    __syncthreads();
    uint2* __restrict__ out = rec + mq.rec + l0;
    for (int x = tid; x < cnt; x += kDrawThreads) out[x] = srec[sord[x]];
    __syncthreads();   // the buffers are reused by the next chunk
  }
  if (bad) atomicOr(&p.sc->err, DERR_SEARCH);
}

// Shared words of the threshold search.
struct PickState {
  alignas(16) uint32_t hist[kBins];
  uint32_t warp_sum[32];
  uint32_t total, bin, above, in_bin;
};

// The highest bin whose count from the top, `above` included, reaches need:
// left in st->bin, with the count above it in st->above and its own in
// st->in_bin.  Every thread of the block (a multiple of 32, at most 1024).
__device__ void pick_bin(PickState* st, uint32_t need, uint32_t above) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = kBins / (int)blockDim.x;
  uint32_t mine = 0;
  for (int x = 0; x < per; ++x) mine += st->hist[kBins - 1 - (tid * per + x)];
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) st->warp_sum[warp] = inc;
  __syncthreads();
  uint32_t before = above + inc - mine;
  for (int w = 0; w < warp; ++w) before += st->warp_sum[w];
  if (before < need && before + mine >= need) {
    for (int x = 0; x < per; ++x) {
      const uint32_t v = st->hist[kBins - 1 - (tid * per + x)];
      if (before + v >= need) {
        st->bin = (uint32_t)(kBins - 1 - (tid * per + x));
        st->above = before;
        st->in_bin = v;
        break;
      }
      before += v;
    }
  }
  __syncthreads();
}

// A threshold (xt, njt): the elements with x > xt, or x == xt and ~j >= njt,
// hold the `need` first by (x desc, j asc) and are at most cap (> need).
// get(e, &x, &j) is element e < n, false where there is none (or x <= 0).
// First the logarithmic bucket of x (16 to an octave: for a few hundred of
// several thousand that is mostly enough), then digits of 11 bits below it, then
// of ~j among equal x; the search ends as soon as the ties of the last step
// fit, and the composite is distinct, so it always ends.  Every thread of the
// block.
template <typename Get>
__device__ void find_threshold(PickState* st, int n, uint32_t need, uint32_t cap, Get get,
                               unsigned long long* xt, uint32_t* njt) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) st->total = 0;
  for (int b = tid; b < kBins; b += blockDim.x) st->hist[b] = 0;
  __syncthreads();
  uint32_t cnt = 0;
  for (int e = tid; e < n; e += blockDim.x) {
    unsigned long long x;
    uint32_t j;
    if (get(e, &x, &j)) {
      ++cnt;
      atomicAdd(&st->hist[log_bucket(x)], 1u);
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
  if (lane == 0 && cnt) atomicAdd(&st->total, cnt);
  __syncthreads();
  *xt = 1;
  *njt = 0;
  if (st->total <= cap) {
    __syncthreads();
    return;
  }
  pick_bin(st, need, 0);
  const uint32_t b0 = st->bin;
  uint32_t above = st->above;
  const uint32_t in_b0 = st->in_bin;
  __syncthreads();
  if (above + in_b0 <= cap) {
    *xt = bucket_floor(b0);
    return;
  }
  // The bucket's values share their leading bits: the exponent's and four more.
  const int ex = (int)(b0 >> 4);
  int top = ex >= 4 ? ex - 4 : 0;                      // bits of x not yet fixed
  unsigned long long prefix = bucket_floor(b0) >> top;  // x >> top of the threshold
  while (top > 0) {
    const int width = top < 11 ? top : 11, sh = top - width;
    for (int b = tid; b < kBins; b += blockDim.x) st->hist[b] = 0;
    __syncthreads();
    for (int e = tid; e < n; e += blockDim.x) {
      unsigned long long x;
      uint32_t j;
      if (get(e, &x, &j) && (top >= 64 || (x >> top) == prefix))
        atomicAdd(&st->hist[(uint32_t)(x >> sh) & ((1u << width) - 1u)], 1u);
    }
    __syncthreads();
    pick_bin(st, need, above);
    prefix = (prefix << width) | st->bin;
    above = st->above;
    const uint32_t in_bin = st->in_bin;
    top = sh;
    __syncthreads();
    if (above + in_bin <= cap) {
      *xt = prefix << top;
      *xt = *xt ? *xt : 1ull;
      return;
    }
  }
  *xt = prefix;
  uint32_t np = 0;
  int ntop = 32;
  while (ntop > 0) {   // ties of x: the smallest j
    const int width = ntop < 11 ? ntop : 11, sh = ntop - width;
    for (int b = tid; b < kBins; b += blockDim.x) st->hist[b] = 0;
    __syncthreads();
    for (int e = tid; e < n; e += blockDim.x) {
      unsigned long long x;
      uint32_t j;
      if (get(e, &x, &j) && x == prefix && (ntop >= 32 || (~j >> ntop) == np))
        atomicAdd(&st->hist[(~j >> sh) & ((1u << width) - 1u)], 1u);
    }
    __syncthreads();
    pick_bin(st, need, above);
    np = (np << width) | st->bin;
    above = st->above;
    const uint32_t in_bin = st->in_bin;
    ntop = sh;
    __syncthreads();
    if (above + in_bin <= cap) break;
  }
  *njt = np << ntop;
}

// A kept column: its x and j.
struct Kept {
  unsigned long long x, j;
};

// Step 2: part u - ubase of query unit_q[u].  The table is open addressing
// with linear probing over 32-bit columns; the sums are 64-bit (two 32-bit
// shared atomics, the low word's carry into the high word).  When it fills up
// (a statistical rarity, or every part of a batch whose parts are capped at
// kMaxParts) the part is taken in 2, 4, ... slices of another mix of j, each
// slice's kept columns competing with those of the slices before.  Once one
// record has found no slot, the others are left: with each of them looking for a
// free slot through the whole table, one query of 8e7 diamonds on 4e7 items took
// 627 ms, 35 so.
//
// The part's records lie in one run per chunk of the query: the runs' offsets are
// scanned (kGroup chunks at a time) and the records dealt out evenly, four of a
// lane read at a time.  Bound by the instructions of the inserts (62 % of the issue
// slots with the loads' latency hidden): a warp that probes until the last of its
// records is placed takes eight to ten steps for two on average, so a record whose
// first slot is taken (a third of them) waits in the warp's queue until 32
// such can probe on together: 14.5 ms for 5e8 diamonds, 9.6 so (four slots per
// load 14.6, four records probing side by side 13.7).
__global__ void __launch_bounds__(kPartThreads, 2)
k_mips_parts(const MipsQuery* __restrict__ queries, const uint32_t* __restrict__ unit_q,
             const uint2* __restrict__ rec, const uint16_t* __restrict__ off, int chunk,
             int slots_max, float factor, int f_exp, uint32_t tprime, Kept* __restrict__ kept,
             uint32_t* __restrict__ kept_n, DevScalars* sc) {
  extern __shared__ __align__(16) unsigned char part_smem[];
  unsigned long long* vals = (unsigned long long*)part_smem;   // slots_max sums
  Kept* temp = (Kept*)(vals + slots_max);                      // cap kept columns
  __shared__ PickState pick;
  __shared__ uint32_t s_full, s_n;
  __shared__ unsigned long long s_inserted, s_created;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kPartThreads / 32;
  const uint32_t u = blockIdx.x;
  const uint32_t q = __ldg(unit_q + u);
  const MipsQuery mq = queries[q];
  const uint32_t part = u - mq.ubase;
  uint32_t* keys = (uint32_t*)(temp + mq.cap);
  const uint32_t cap = mq.cap;
  Kept* __restrict__ list = kept + mq.cand + (unsigned long long)part * cap;
  const uint32_t nch = (uint32_t)((mq.s + chunk - 1) / chunk);
  const uint16_t* __restrict__ o = off + mq.off + part;
  const uint32_t ostep = mq.parts + 1;
  // Chunks g0 .. of the part: soff[c] the records of those before chunk g0 + c,
  // srun[c] + e the place of record e of them after chunk g0's first record;
  // returns how many they are.
  __shared__ uint32_t soff[kGroup], srun[kGroup];
  uint2* queue = (uint2*)pick.hist + 64 * warp;
  auto scan_group = [&](uint32_t g0) -> uint32_t {
    const uint32_t c = g0 + tid;
    uint32_t b0 = 0, len = 0;
    if (c < nch) {
      b0 = __ldg(o + (size_t)c * ostep);
      len = (uint32_t)__ldg(o + (size_t)c * ostep + 1) - b0;
    }
    uint32_t inc = len;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, inc, s);
      if (lane >= s) inc += v;
    }
    __syncthreads();   // (the words may still be read)
    if (lane == 31) pick.warp_sum[warp] = inc;
    __syncthreads();
    uint32_t before = inc - len, total = 0;
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t v = pick.warp_sum[w];
      before += w < warp ? v : 0u;
      total += v;
    }
    soff[tid] = before;
    srun[tid] = (uint32_t)tid * (uint32_t)chunk + b0 - before;
    __syncthreads();
    return total;
  };
  unsigned long long records = 0;
  uint32_t in_group = 0;
  for (uint32_t g0 = 0; g0 < nch; g0 += kGroup) records += in_group = scan_group(g0);
  // A power of two of at least `factor` slots per record (1.5 unless a test
  // asks for less), up to the table's size.
  int slots = 256;
  while (slots < slots_max && (float)slots < factor * (float)records) slots <<= 1;
  const uint32_t mask = (uint32_t)slots - 1;
  for (int level = 0; level <= 31; ++level) {
    uint32_t nlist = 0;
    bool full = false;
    if (tid == 0) s_inserted = s_created = 0;
    const uint32_t slices = 1u << level;
    for (uint32_t slice = 0; slice < slices && !full; ++slice) {
      for (int x = tid; x < slots / 4; x += kPartThreads)
        ((uint4*)keys)[x] = make_uint4(kNoKey, kNoKey, kNoKey, kNoKey);
      for (int x = tid; x < slots / 2; x += kPartThreads)
        ((uint4*)vals)[x] = make_uint4(0u, 0u, 0u, 0u);
      if (tid == 0) s_full = 0;
      __syncthreads();
      unsigned long long ins = 0, cre = 0;
      auto add = [&](uint32_t slot, long long x) {
        uint32_t* h2 = (uint32_t*)(vals + slot);
        const uint32_t lo = (uint32_t)(unsigned long long)x;
        const uint32_t hi = (uint32_t)((unsigned long long)x >> 32);
        const uint32_t old = atomicAdd(h2, lo);
        atomicAdd(h2 + 1, hi + (old + lo < old ? 1u : 0u));
      };
      // The slots after its first, of a record that found that taken.
      auto probe_on = [&](uint2 v) {
        uint32_t slot = fmix32(v.x) & mask;
        int probes = 1;
        for (; probes < slots; ++probes) {
          if ((probes & 63) == 0 && *(volatile uint32_t*)&s_full) break;
          slot = (slot + 1) & mask;
          const uint32_t cur = atomicCAS(keys + slot, kNoKey, v.x);
          if (cur == kNoKey || cur == v.x) {
            cre += cur == kNoKey ? 1 : 0;
            add(slot, fixed_point(__uint_as_float(v.y), f_exp));
            break;
          }
        }
        if (probes == slots) s_full = 1;
      };
      int waiting = 0;   // of the warp
      for (uint32_t g0 = 0; g0 < nch; g0 += kGroup) {
        if (nch > (uint32_t)kGroup) {
          if (g0 && __syncthreads_or((int)s_full)) break;
          in_group = scan_group(g0);
        }
        const int runs = (int)(nch - g0 < (uint32_t)kGroup ? nch - g0 : (uint32_t)kGroup);
        const uint2* __restrict__ r = rec + mq.rec + (unsigned long long)g0 * chunk;
        // A warp's records: an even share of them, in a row.
        const uint32_t share = ((in_group + kPartThreads - 1) / kPartThreads) * 32;
        const uint32_t end = min(in_group, (warp + 1) * share);
        int run = 0;   // the last run that starts at or before the lane's record
        for (uint32_t base = warp * share; base < end; base += 32 * kAhead) {
          if (__any_sync(0xFFFFFFFFu, *(volatile uint32_t*)&s_full)) break;
          uint2 v[kAhead];
#pragma unroll
          for (int a = 0; a < kAhead; ++a) {
            const uint32_t e = base + 32 * a + lane;
            v[a] = make_uint2(0u, 0u);
            if (e < end) {
              if (run + 1 < runs && soff[run + 1] <= e) {
                ++run;
                if (run + 1 < runs && soff[run + 1] <= e)
                  for (int step = 1 << (31 - __clz(runs)); step > 0; step >>= 1)
                    if (run + step < runs && soff[run + step] <= e) run += step;
              }
              v[a] = __ldg(r + (uint32_t)(srun[run] + e));
            }
          }
#pragma unroll
          for (int a = 0; a < kAhead; ++a) {
            const long long x = fixed_point(__uint_as_float(v[a].y), f_exp);   // (0: no record)
            const uint32_t h = fmix32(v[a].x), slot = h & mask;
            const bool in = x != 0 && !(level && (fmix32(h ^ 0x9E3779B9u) >> (32 - level)) != slice);
            bool wait = false;
            if (in) {
              ++ins;
              const uint32_t cur = atomicCAS(keys + slot, kNoKey, v[a].x);
              if (cur == kNoKey || cur == v[a].x) {
                cre += cur == kNoKey ? 1 : 0;
                add(slot, x);
              } else {
                wait = true;
              }
            }
            const uint32_t left = __ballot_sync(0xFFFFFFFFu, wait);
            if (left) {
              if (wait) queue[waiting + __popc(left & ((1u << lane) - 1u))] = v[a];
              waiting += __popc(left);
              __syncwarp();
              if (waiting >= 32) {
                waiting -= 32;
                probe_on(queue[waiting + lane]);
                __syncwarp();
              }
            }
          }
        }
      }
      if (lane < waiting) probe_on(queue[lane]);
#pragma unroll
      for (int s = 16; s >= 1; s >>= 1) {
        ins += __shfl_xor_sync(0xFFFFFFFFu, ins, s);
        cre += __shfl_xor_sync(0xFFFFFFFFu, cre, s);
      }
      if (lane == 0) {
        if (ins) atomicAdd(&s_inserted, ins);
        if (cre) atomicAdd(&s_created, cre);
      }
      if (tid == 0) s_n = 0;
      __syncthreads();
      full = s_full != 0;
      if (full) {
        __syncthreads();
        break;
      }
      auto get = [&](int e, unsigned long long* x, uint32_t* j) {
        if (e < slots) {
          *x = vals[e];
          if ((long long)*x <= 0) return false;   // (0 in a free slot)
          *j = keys[e];
          return true;
        }
        const Kept k = list[e - slots];
        *x = k.x;
        *j = (uint32_t)k.j;
        return true;
      };
      unsigned long long xt;
      uint32_t njt;
      const int n = slots + (int)nlist;
      find_threshold(&pick, n, tprime, cap, get, &xt, &njt);
      for (int e = tid; e < n; e += kPartThreads) {
        unsigned long long x;
        uint32_t j;
        if (get(e, &x, &j) && (x > xt || (x == xt && ~j >= njt))) {
          const uint32_t at = atomicAdd(&s_n, 1u);
          if (at < cap) {
            temp[at].x = x;
            temp[at].j = j;
          }
        }
      }
      __syncthreads();
      nlist = s_n < cap ? s_n : cap;
      for (uint32_t e = tid; e < nlist; e += kPartThreads) list[e] = temp[e];
      __syncthreads();
    }
    if (!full) {
      if (tid == 0) {
        kept_n[u] = nlist;
        if (s_inserted) atomicAdd(&sc->inserted, s_inserted);
        if (s_created) atomicAdd(&sc->new_keys, s_created);
      }
      return;
    }
  }
  if (tid == 0) {   // (not reached: 2^31 slices hold two columns each)
    kept_n[u] = 0;
    atomicOr(&sc->err, DERR_HASH_FULL);
  }
}

// Bitonic sort of n (a power of two, <= kSortMax) entries of shared arrays
// into "before" order; all threads of the block take part.
template <typename Before>
__device__ void block_bitonic(unsigned long long* a, unsigned long long* b, double* c, int n,
                              Before before) {
  for (int k = 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
        const int x = ((t & ~(j - 1)) << 1) | (t & (j - 1)), y = x + j;   // j a power of two
        const bool up = (x & k) == 0;
        const bool y_first = before(a[y], b[y], c ? c[y] : 0.0, a[x], b[x], c ? c[x] : 0.0);
        if (y_first == up) {
          const unsigned long long ta = a[x], tb = b[x];
          a[x] = a[y]; b[x] = b[y]; a[y] = ta; b[y] = tb;
          if (c) {
            const double tc = c[x];
            c[x] = c[y];
            c[y] = tc;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Step 3, query blockIdx.x: the t' first of its parts' kept columns by (x
// desc, j asc), sorted; then c = q . b_j in FP64 (32 lane-strided fused
// multiply-add partial sums folded in halves) and the t largest |c| by (|c|
// desc, j asc).
__global__ void __launch_bounds__(512)
k_mips_final(const MipsQuery* __restrict__ queries, const Kept* __restrict__ kept,
             const uint32_t* __restrict__ kept_n, const float* __restrict__ Q, int64_t ldq,
             const float* __restrict__ Bt, int64_t d, uint32_t tprime, uint32_t t,
             mad_pair* __restrict__ out, uint32_t* __restrict__ nout,
             mad_pair* __restrict__ cand_out) {
  __shared__ unsigned long long cx[kSortMax], ck[kSortMax];
  __shared__ PickState pick;
  static_assert(kTPrimeMax * sizeof(double) <= kBins * sizeof(uint32_t), "c in the bins' place");
  double* cc = (double*)pick.hist;   // (the search is over when the t' are rescored)
  __shared__ uint32_t s_n;
  const uint32_t q = blockIdx.x;
  const MipsQuery mq = queries[q];
  const Kept* __restrict__ list = kept + mq.cand;
  const uint32_t* __restrict__ cnt = kept_n + mq.ubase;
  auto get = [&](int e, unsigned long long* x, uint32_t* j) {
    const uint32_t part = (uint32_t)e / mq.cap;
    if ((uint32_t)e - part * mq.cap >= __ldg(cnt + part)) return false;
    const Kept k = list[e];
    *x = k.x;
    *j = (uint32_t)k.j;
    return true;
  };
  const int total = (int)(mq.parts * mq.cap);
  unsigned long long xt = 1;
  uint32_t njt = 0;
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  const uint32_t cap = min((uint32_t)kSortMax, tprime + (uint32_t)kSlack);
  if (mq.parts > 1) find_threshold(&pick, total, tprime, cap, get, &xt, &njt);
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    unsigned long long x;
    uint32_t j;
    if (get(e, &x, &j) && (x > xt || (x == xt && ~j >= njt))) {
      const uint32_t at = atomicAdd(&s_n, 1u);
      if (at < kSortMax) {
        cx[at] = x;
        ck[at] = j;
      }
    }
  }
  __syncthreads();
  const int n = (int)min(s_n, (uint32_t)kSortMax);
  int n2 = 1;
  while (n2 < n) n2 <<= 1;
  for (int x = n + threadIdx.x; x < n2; x += blockDim.x) {
    cx[x] = 0;           // sorts after every collected x (all positive)
    ck[x] = ~0ull;
  }
  __syncthreads();
  block_bitonic(cx, ck, (double*)nullptr, n2,
                [](unsigned long long ax, unsigned long long ak, double, unsigned long long bx,
                   unsigned long long bk, double) { return ax > bx || (ax == bx && ak < bk); });
  const int K = n < (int)tprime ? n : (int)tprime;
  if (cand_out) {
    for (int x = threadIdx.x; x < K; x += blockDim.x) {
      mad_pair pr;
      pr.i = q;
      pr.j = (uint32_t)ck[x];
      pr.x = (int64_t)cx[x];
      pr.c = 0.0;
      cand_out[(size_t)q * tprime + x] = pr;
    }
  }
  // Exact rescoring, one warp per candidate; when t is a small part of K, only
  // of the candidates that FP32 bounds leave (as k_rescore_bound: FP64 runs at
  // a sixty-fourth of FP32, and t' = 100 products of d = 300 cost a query 12 us
  // of it): a candidate whose U lies below t others' L is not among the t largest.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const float* __restrict__ a = Q + (int64_t)q * ldq;
  static_assert(kSortMax >= 2 * kTPrimeMax, "bounds in the upper half of cx");
  float2* lu = (float2*)(cx + kTPrimeMax);
  const bool bounded = 4 * (int)t <= K;
  if (bounded) {
    for (int x = warp; x < K; x += warps) {
      const float* __restrict__ b = Bt + (int64_t)(uint32_t)ck[x] * d;
      float c = 0.0f, s = 0.0f;
      for (int64_t k = lane; k < d; k += 32) {
        c = fmaf(a[k], b[k], c);
        s = fmaf(fabsf(a[k]), fabsf(b[k]), s);
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) {
        c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      }
      if (lane == 0) {
        const float inf = __int_as_float(0x7F800000);
        const bool known = s < inf && fabsf(c) < inf;
        const float e = fmaf(s, kBoundEps, kBoundTiny);
        lu[x] = known ? make_float2(fabsf(c) - e, fabsf(c) + e) : make_float2(0.0f, inf);
      }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < K; x += blockDim.x) {
      const float up = lu[x].y;
      int over = 0;
      for (int y = 0; y < K; ++y) over += lu[y].x > up ? 1 : 0;
      if (over >= (int)t) ck[x] = ~0ull;   // sorts last, as a padding entry
    }
    __syncthreads();
  }
  for (int x = warp; x < K; x += warps) {
    if (ck[x] == ~0ull) {
      if (lane == 0) cc[x] = -1.0;
      continue;
    }
    const float* __restrict__ b = Bt + (int64_t)(uint32_t)ck[x] * d;
    double acc = 0.0;
    for (int64_t k = lane; k < d; k += 32) acc = __fma_rn((double)a[k], (double)b[k], acc);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, off));
    if (lane == 0) cc[x] = acc;
  }
  __syncthreads();
  // The t largest |c| among the K: sort the K by (|c| desc, key asc).
  int k2 = 1;
  while (k2 < K) k2 <<= 1;
  for (int x = K + threadIdx.x; x < k2; x += blockDim.x) {
    cx[x] = 0;
    ck[x] = ~0ull;
    cc[x] = -1.0;   // |c| of a padding entry is below every real |c|
  }
  __syncthreads();
  if (K > 1)
    block_bitonic(cx, ck, cc, k2,
                  [](unsigned long long, unsigned long long ak, double ac, unsigned long long,
                     unsigned long long bk, double bc) {
                    const double fa = ac < 0.0 && ak == ~0ull ? -1.0 : fabs(ac);
                    const double fb = bc < 0.0 && bk == ~0ull ? -1.0 : fabs(bc);
                    return fa > fb || (fa == fb && ak < bk);
                  });
  const int T = K < (int)t ? K : (int)t;
  for (int x = threadIdx.x; x < T; x += blockDim.x) {
    mad_pair pr;
    pr.i = q;
    pr.j = (uint32_t)ck[x];
    pr.x = (int64_t)cx[x];
    pr.c = cc[x];
    out[(size_t)q * t + x] = pr;
  }
  if (threadIdx.x == 0) nout[q] = (uint32_t)T;
}

template <typename T>
mad_status pool_alloc(mad_ctx* ctx, T*& p, size_t count, cudaStream_t st) {
  if (count == 0) count = 1;
  void* q = nullptr;
  const mad_status rs = pool_malloc(ctx, &q, count * sizeof(T), st);
  p = (T*)q;
  return rs;
}

template <typename T>
void pool_free(T*& p, cudaStream_t st) {
  if (p) cudaFreeAsync((void*)p, st);
  p = nullptr;
}

// A part's table, its kept columns and the columns' keys.
size_t parts_smem_bytes(int slots, uint32_t cap) {
  return (size_t)slots * 12 + (size_t)cap * sizeof(Kept);
}

// The batch's device buffer: the queries, the query of every chunk and part,
// the part offsets of every chunk, the records and the parts' kept columns.
struct MipsBufs {
  MipsQuery* queries;
  uint32_t* chunk_q;
  uint32_t* unit_q;
  uint16_t* off;
  uint2* rec;
  Kept* kept;
  uint32_t* kept_n;
  size_t bytes;
};

MipsBufs carve_mips(void* base, uint64_t nq, uint64_t chunks, uint64_t units, uint64_t offs,
                    uint64_t records, uint64_t kept) {
  MipsBufs b;
  char* p = (char*)base;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char* q = p ? p + at : nullptr;
    at += (bytes + 255) & ~(size_t)255;
    return (void*)q;
  };
  b.queries = (MipsQuery*)take(nq * sizeof(MipsQuery));
  b.chunk_q = (uint32_t*)take(chunks * sizeof(uint32_t));
  b.unit_q = (uint32_t*)take(units * sizeof(uint32_t));
  b.off = (uint16_t*)take(offs * sizeof(uint16_t));
  b.rec = (uint2*)take(records * sizeof(uint2));
  b.kept = (Kept*)take(kept * sizeof(Kept));
  b.kept_n = (uint32_t*)take(units * sizeof(uint32_t));
  b.bytes = at;
  return b;
}

}  // namespace
}  // namespace mad

using namespace mad;

extern "C" {

mad_status mad_mips_items(mad_ctx* ctx, const mad_matrix* B, uint64_t s_max, mad_stream stream) {
  if (!ctx || !B || s_max == 0 || s_max > (1ull << 40)) return MAD_ERR_ARG;
  if (B->fmt != MAD_DENSE_ROWMAJOR || B->dt != MAD_F32 || !B->values || B->rows <= 0 ||
      B->cols <= 0 || B->ld < B->cols)
    return MAD_ERR_ARG;
  if (B->cols >= (1ll << 31) || B->rows > kItemDimMax) return MAD_ERR_UNSUPPORTED;
  if (ctx->flags) return MAD_ERR_UNSUPPORTED;   // plain |q . b_j|, no Gram or sign flags
  cudaStream_t st = (cudaStream_t)stream;
  cudaStreamSynchronize(st);
  // Drop every earlier table (single-instance or batched).
  pool_free(ctx->T1, st); pool_free(ctx->T2, st); pool_free(ctx->TA, st); pool_free(ctx->TB, st);
  pool_free(ctx->na, st); pool_free(ctx->nb, st); pool_free(ctx->r, st); pool_free(ctx->r64, st);
  pool_free(ctx->bt, st); pool_free(ctx->hkeys, st); pool_free(ctx->hvals, st);
  pool_free(ctx->hreg, st); pool_free(ctx->T2g_ptr, st);
  pool_free(ctx->T2g, st); pool_free(ctx->T2g_sh, st); pool_free(ctx->bloom, st);
  pool_free(ctx->TBg, st); pool_free(ctx->TBg_sh, st);
  pool_free(ctx->mips_buf, st); pool_free(ctx->tb_row, st);
  pool_free(ctx->tb_blocks, st);
  pool_free(ctx->pipe_buf, st);
  pool_free(ctx->pipe_scratch, st);
  ctx->pipe_scratch_bytes = 0;
  ctx->pipe = false;
  ctx->built = false;
  ctx->mips_items = false;
  ctx->shape.valid = false;
  ctx->mips_nq = 0;
  ctx->B = *B;
  ctx->dense = true;
  ctx->integer = false;
  ctx->regioned = true;
  ctx->hov = 0;
  ctx->d = B->rows;
  ctx->n = B->cols;
  ctx->m = 0;
  ctx->s_max = s_max;
  mad_status rs;
  if ((rs = pool_alloc(ctx, ctx->TB, (size_t)(ctx->d * ctx->n) + 4, st)) != MAD_OK) return rs;
  if ((rs = pool_alloc(ctx, ctx->nb, (size_t)ctx->d, st)) != MAD_OK) return rs;
  char* bt = nullptr;
  if ((rs = pool_alloc(ctx, bt, (size_t)(ctx->n * ctx->d) * 4, st)) != MAD_OK) return rs;
  ctx->bt = bt;
  // (a test asks for the guides by an overflow table of the debug layout)
  if (ctx->hov_request == 0 && tb_blocks_apply(ctx->d, ctx->n)) {
    if ((rs = pool_alloc(ctx, ctx->tb_row, (size_t)ctx->d, st)) != MAD_OK) return rs;
    if ((rs = pool_alloc(ctx, ctx->tb_blocks, tb_blocks_quads(ctx->d, ctx->n), st)) != MAD_OK)
      return rs;
  } else {
    ctx->tbg_stride = ((int64_t)1 << tb_guide_width(ctx->n)) + 1;
    if ((rs = pool_alloc(ctx, ctx->TBg_sh, (size_t)ctx->d, st)) != MAD_OK) return rs;
    if ((rs = pool_alloc(ctx, ctx->TBg, (size_t)(ctx->d * ctx->tbg_stride), st)) != MAD_OK)
      return rs;
  }
  cudaMemsetAsync(ctx->sc, 0, sizeof(DevScalars), st);
  if ((rs = build_item_tables(ctx, st)) != MAD_OK) return rs;
  if ((rs = tb_guide_build(ctx, st)) != MAD_OK) return rs;
  DevScalars hs;
  cudaMemcpyAsync(&hs, ctx->sc, sizeof(hs), cudaMemcpyDeviceToHost, st);
  if ((rs = cuda_status(cudaStreamSynchronize(st))) != MAD_OK) return rs;
  if (hs.maxb_bits == 0u) return MAD_ERR_EMPTY;
  float maxb;
  std::memcpy(&maxb, &hs.maxb_bits, sizeof(float));
  int lgs = 0;
  while (lgs < 64 && (1ull << lgs) < s_max) ++lgs;
  ctx->f = 62 - lgs - (std::ilogb(maxb) + 1);
  ctx->mips_items = true;
  return cuda_status(cudaStreamSynchronize(st));
}

mad_status mad_mips_config(mad_ctx* ctx, uint32_t region_lg, uint32_t chunk_mult,
                           uint32_t blocks_per_sm, uint32_t select_threads) {
  if (!ctx || region_lg > 4 || blocks_per_sm > 8) return MAD_ERR_ARG;
  if (chunk_mult != 0 && chunk_mult != 1 && chunk_mult != 2 && chunk_mult != 4 && chunk_mult != 8)
    return MAD_ERR_ARG;
  if (select_threads != 0 && select_threads != 128 && select_threads != 256 &&
      select_threads != 512)
    return MAD_ERR_ARG;
  ctx->mips_region_lg = region_lg == 0 ? 1 : (int)region_lg;
  ctx->mips_chunk_mult = chunk_mult == 0 ? 8 : (int)chunk_mult;
  ctx->mips_bps = (int)blocks_per_sm;
  ctx->mips_select_threads = select_threads == 0 ? 256 : (int)select_threads;
  return MAD_OK;
}

mad_status mad_mips_plan(mad_ctx* ctx, uint32_t nq, const uint64_t* s_host, uint32_t tprime,
                         uint32_t t, mad_stream stream) {
  if (!ctx || !s_host || nq == 0 || tprime == 0 || tprime > (uint32_t)kTPrimeMax || t == 0 ||
      t > tprime)
    return MAD_ERR_ARG;
  if (!ctx->mips_items) return MAD_ERR_STATE;
  cudaStream_t st = (cudaStream_t)stream;
  const uint64_t chunk = (uint64_t)kDrawThreads * (uint64_t)ctx->mips_chunk_mult;
  // Distinct columns a part's table is planned for: load 0.6 at region_lg =
  // 1, half of it for each step above.
  const uint64_t part_keys = (uint64_t)(kSlots * 6 / 10) >> (ctx->mips_region_lg - 1);
  std::vector<MipsQuery> qs(nq);
  uint64_t chunks = 0, units = 0, offs = 0, records = 0, kept = 0, most = 0;
  uint32_t max_parts = 1, max_cap = 1;
  for (uint32_t q = 0; q < nq; ++q) {
    const uint64_t s = s_host[q];
    if (s == 0 || s > ctx->s_max) return MAD_ERR_ARG;
    const uint64_t distinct = std::min<uint64_t>(s, (uint64_t)ctx->n);
    const uint64_t nch = (s + chunk - 1) / chunk;
    MipsQuery& m = qs[q];
    m.s = s;
    m.rec = records;
    m.off = offs;
    m.cand = kept;
    m.parts = (uint32_t)std::min<uint64_t>(kMaxParts, (distinct + part_keys - 1) / part_keys);
    m.ubase = (uint32_t)units;
    m.cbase = (uint32_t)chunks;
    m.cap = (uint32_t)std::min<uint64_t>(distinct, (uint64_t)tprime + kSlack);
    chunks += nch;
    units += m.parts;
    offs += nch * (m.parts + 1);
    records += s;
    kept += (uint64_t)m.parts * m.cap;
    most = std::max(most, (distinct + m.parts - 1) / m.parts);
    max_parts = std::max(max_parts, m.parts);
    max_cap = std::max(max_cap, m.cap);
    // (a batch this long holds tens of terabytes of records)
    if (chunks >= (1ull << 32) || units >= (1ull << 31)) return MAD_ERR_OOM;
  }
  std::vector<uint32_t> cq, uq;
  cq.reserve(chunks);
  uq.reserve(units);
  for (uint32_t q = 0; q < nq; ++q) {
    cq.insert(cq.end(), (size_t)((qs[q].s + chunk - 1) / chunk), q);
    uq.insert(uq.end(), qs[q].parts, q);
  }
  cudaStreamSynchronize(st);
  pool_free(ctx->T2, st); pool_free(ctx->TA, st); pool_free(ctx->na, st); pool_free(ctx->r, st);
  pool_free(ctx->mips_buf, st);
  ctx->mips_nq = 0;
  mad_status rs;
  if ((rs = pool_alloc(ctx, ctx->T2, (size_t)nq * (size_t)ctx->d, st)) != MAD_OK) return rs;
  if ((rs = pool_alloc(ctx, ctx->TA, (size_t)nq * (size_t)ctx->d, st)) != MAD_OK) return rs;
  if ((rs = pool_alloc(ctx, ctx->na, (size_t)nq, st)) != MAD_OK) return rs;
  if ((rs = pool_alloc(ctx, ctx->r, (size_t)nq, st)) != MAD_OK) return rs;
  const MipsBufs sizes = carve_mips(nullptr, nq, chunks, units, offs, records, kept);
  if ((rs = pool_malloc(ctx, &ctx->mips_buf, sizes.bytes, st)) != MAD_OK) return rs;
  const MipsBufs b = carve_mips(ctx->mips_buf, nq, chunks, units, offs, records, kept);
  cudaMemcpyAsync(b.queries, qs.data(), nq * sizeof(MipsQuery), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(b.chunk_q, cq.data(), chunks * sizeof(uint32_t), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(b.unit_q, uq.data(), units * sizeof(uint32_t), cudaMemcpyHostToDevice, st);
  if ((rs = cuda_status(cudaStreamSynchronize(st))) != MAD_OK) return rs;
  int slots = 256;   // the largest table any part starts with
  while (slots < kSlots && (uint64_t)slots * 2 < most * 3) slots <<= 1;
  ctx->m = nq;
  ctx->hcap = ctx->hcap_alloc = 0;
  ctx->mips_nq = nq;
  ctx->mips_tprime = tprime;
  ctx->mips_t = t;
  ctx->mips_chunks = chunks;
  ctx->mips_units = units;
  ctx->mips_offs = offs;
  ctx->mips_records = records;
  ctx->mips_kept = kept;
  ctx->mips_max_parts = max_parts;
  ctx->mips_slots = slots;
  ctx->mips_parts_smem = parts_smem_bytes(slots, max_cap);
  ctx->mips_plan_mult = ctx->mips_chunk_mult;
  cudaError_t e = cudaFuncSetAttribute(k_mips_draw<true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDrawSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mips_draw<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kDrawSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mips_parts, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)parts_smem_bytes(kSlots, kTPrimeMax + kSlack));
  if (e != cudaSuccess) ctx->mips_nq = 0;   // no plan: a run is refused
  return cuda_status(e);
}

mad_status mad_mips_run(mad_ctx* ctx, const mad_matrix* Q, uint64_t seed, mad_pair* out_dev,
                        uint32_t* n_out_dev, mad_pair* cand_dev, mad_stream stream) {
  if (!ctx || !Q || !out_dev || !n_out_dev) return MAD_ERR_ARG;
  if (!ctx->mips_items || ctx->mips_nq == 0) return MAD_ERR_STATE;
  if (Q->fmt != MAD_DENSE_ROWMAJOR || Q->dt != MAD_F32 || !Q->values ||
      Q->rows != (int64_t)ctx->mips_nq || Q->cols != ctx->d || Q->ld < Q->cols)
    return MAD_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ctx->A = *Q;
  // Query rows of the tables (T2, TA; T1 is not needed: m = 1 per query).
  mad_status rs;
  if ((rs = build_query_rows(ctx, st)) != MAD_OK) return rs;
  const MipsBufs b = carve_mips(ctx->mips_buf, ctx->mips_nq, ctx->mips_chunks, ctx->mips_units,
                                ctx->mips_offs, ctx->mips_records, ctx->mips_kept);
  const SampleParams p = make_params(ctx);
  const int chunk = kDrawThreads * ctx->mips_plan_mult;
  unsigned long long grid = ctx->mips_chunks;
  if (ctx->mips_bps > 0) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = std::min<unsigned long long>(grid, (unsigned long long)sms * ctx->mips_bps);
  }
  grid = std::min<unsigned long long>(grid, 0x7FFFFFFFull);
  const size_t draw_smem = draw_smem_bytes(chunk, ctx->mips_max_parts, ctx->d);
  if (p.tb_blocks)
    k_mips_draw<true><<<(unsigned)grid, kDrawThreads, draw_smem, st>>>(
        p, seed, b.queries, b.chunk_q, ctx->mips_chunks, ctx->mips_plan_mult, ctx->mips_max_parts,
        b.rec, b.off);
  else
    k_mips_draw<false><<<(unsigned)grid, kDrawThreads, draw_smem, st>>>(
        p, seed, b.queries, b.chunk_q, ctx->mips_chunks, ctx->mips_plan_mult, ctx->mips_max_parts,
        b.rec, b.off);
  // The next two kernels read addresses out of what this one writes.
  if ((rs = cuda_status(cudaGetLastError())) != MAD_OK) return rs;
  k_mips_parts<<<(unsigned)ctx->mips_units, kPartThreads, ctx->mips_parts_smem, st>>>(
      b.queries, b.unit_q, b.rec, b.off, chunk, ctx->mips_slots, ctx->region_factor, ctx->f, ctx->mips_tprime, b.kept,
      b.kept_n, ctx->sc);
  if ((rs = cuda_status(cudaGetLastError())) != MAD_OK) return rs;
  k_mips_final<<<ctx->mips_nq, ctx->mips_select_threads, 0, st>>>(
      b.queries, b.kept, b.kept_n, (const float*)Q->values, Q->ld, (const float*)ctx->bt, ctx->d,
      ctx->mips_tprime, ctx->mips_t, out_dev, n_out_dev, cand_dev);
  count_launch(ctx, 3);
  return cuda_status(cudaGetLastError());
}

}  // extern "C"
