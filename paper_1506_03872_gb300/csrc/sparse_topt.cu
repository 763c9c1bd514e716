// Exact comparator for 0/1 inputs: the t largest c_ij of C = A B by direct
// sparse computation (the paper's exact computation for comparison, Sec.
// 4.3, which forms C one sparse vector at a time and keeps the top entries
// in a priority queue), rebuilt for the GPU around a fused threshold.
//
// For 0/1 inputs c_ij counts the k with a_ik = b_kj = 1, so c_ij <=
// min(nnz(a_i*), nnz(b_*j)).  With theta a lower bound on the t-th largest
// entry tau, no row with fewer than theta entries and no column of B with
// fewer than theta entries can hold a pair of the top t, so:
//
//   1. pilot: the exact counts among the rows of A and columns of B of largest
//      degree (16 sqrt(t) of each, 256 to 2048); the t-th largest of them is such a theta (t entries
//      of C are at least that large);
//   2. main pass over the rows with nnz >= theta against the columns with
//      nnz >= theta only: B is filtered to those columns and relabelled by
//      their rank (a monotone map, so every row of B stays sorted), each row
//      i of C is accumulated in shared-memory count windows (one block per
//      row, rows handed out through an atomic counter in decreasing degree
//      order), and its entries with c >= theta go to a candidate list;
//   3. the t largest candidates by (c desc, key asc), sorted.
//
// Entries equal to the t-th value are ties; if the candidates overflow the
// list, the exact tau comes from the histogram of the emitted counts and
// the pass repeats: every c > tau, then the smallest keys among c == tau
// (per-row tie counts, their prefix over rows in index order, and the first
// ties of the boundary row in ascending j).  The result equals the oracle's
// row-wise sparse product for any input.  With MAD_SPARSE_NO_BOUND the main
// pass takes every row and column (only the threshold filters entries).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "mad_internal.cuh"

namespace mad {
namespace {

constexpr int kSpBlock = 512;
constexpr int kSpWarps = kSpBlock / 32;
constexpr uint32_t kSpWindowMax = 24576;       // labels per shared window (96 KB)
// Rows and columns of the pilot: its pairs have to hold t large counts, so its
// side grows with sqrt(t).  16 sqrt(t) measured best between 8 and 64 (2048 at
// t = 1000, the size it always had) on graphs of 2e4 to 1e6 nodes: 1e6 nodes, t
// = 1000: 1224, 1070, 1093, 1098 and 1193 us at 8, 16, 24, 32 and 64 (measured
// side by side).
uint32_t pilot_size(uint32_t t) {
  const double want = 16.0 * std::sqrt((double)t);
  return want < 256.0 ? 256u : want > 2048.0 ? 2048u : (uint32_t)want;
}
constexpr uint32_t kHistSmem = 4096;           // pilot histogram bins (clamped)
constexpr uint32_t kHistGlobal = 65536;        // main-pass histogram bins (clamped)
constexpr uint64_t kSpListCap = 1ull << 20;    // candidate list entries
constexpr unsigned FULL = 0xffffffffu;

struct SpScalars {
  unsigned int bins[2][32];        // log2-degree bucket counts (rows, columns)
  unsigned int cur[2][32];         // scatter cursors
  unsigned long long count;        // candidates emitted (may pass the capacity)
  unsigned int row_next;           // persistent row counter
  unsigned int theta;              // threshold read from a histogram
  unsigned int row_lim, lim_x;     // tie-limited emission
  unsigned long long need;         // ties still to take
  unsigned int err;
  unsigned int pad;
};

__device__ __forceinline__ uint32_t deg_of(const int64_t* ptr, const uint32_t* cnt, uint64_t i) {
  return ptr ? (uint32_t)(ptr[i + 1] - ptr[i]) : cnt[i];
}

// Column counts of B: cb[j] = nnz of column j.
__global__ void k_col_counts(const int32_t* __restrict__ col, uint64_t nnz, uint32_t* cb) {
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz;
       e += (uint64_t)gridDim.x * blockDim.x)
    atomicAdd(&cb[col[e]], 1u);
}

// Row degrees as counts (Gram inputs: the columns of B = A^T are the rows
// of A).
__global__ void k_row_degrees(const int64_t* __restrict__ ptr, uint64_t n, uint32_t* out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = (uint32_t)(ptr[i + 1] - ptr[i]);
}

// Indices with degree >= th, counted per floor(log2(degree)) bucket.
__global__ void k_logbin_count(const int64_t* ptr, const uint32_t* cnt, uint64_t n, uint32_t th,
                               unsigned int* bins) {
  __shared__ unsigned int sb[32];
  if (threadIdx.x < 32) sb[threadIdx.x] = 0;
  __syncthreads();
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t dg = deg_of(ptr, cnt, i);
    if (dg >= th && dg > 0) atomicAdd(&sb[31 - __clz(dg)], 1u);
  }
  __syncthreads();
  if (threadIdx.x < 32 && sb[threadIdx.x]) atomicAdd(&bins[threadIdx.x], sb[threadIdx.x]);
}

// The same indices in decreasing bucket order (any order within a bucket):
// a schedule and a choice of the heaviest rows, not a result.
__global__ void k_logbin_scatter(const int64_t* ptr, const uint32_t* cnt, uint64_t n, uint32_t th,
                                 const unsigned int* bins, unsigned int* cur, uint32_t* order) {
  __shared__ unsigned int off[32];
  if (threadIdx.x < 32) {
    unsigned int s = 0;
    for (int b = 31; b > (int)threadIdx.x; --b) s += bins[b];
    off[threadIdx.x] = s;
  }
  __syncthreads();
  const unsigned lane = threadIdx.x & 31;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t n_up = (n + 31) & ~31ull;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_up; i += stride) {
    const uint32_t dg = i < n ? deg_of(ptr, cnt, i) : 0;
    const bool take = i < n && dg >= th && dg > 0;
    const int b = take ? 31 - __clz(dg) : -1;
    const unsigned peers = __match_any_sync(FULL, b);
    if (take) {
      const unsigned leader = __ffs(peers) - 1;
      unsigned base = 0;
      if (lane == leader) base = atomicAdd(&cur[b], (unsigned)__popc(peers));
      base = __shfl_sync(peers, base, leader);
      order[off[b] + base + __popc(peers & ((1u << lane) - 1))] = (uint32_t)i;
    }
  }
}

__global__ void k_mark_list(const uint32_t* __restrict__ list, uint32_t h, uint32_t* sel) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < h) sel[list[q]] = 1u;
}

__global__ void k_mark_deg(const uint32_t* __restrict__ cb, uint64_t n, uint32_t th, uint32_t* sel) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (uint64_t)gridDim.x * blockDim.x)
    sel[j] = (cb[j] >= th && cb[j] > 0) ? 1u : 0u;
}

// colmap: the selected columns in order; bits: the selection as a bitmap.
__global__ void k_colmap(const uint32_t* __restrict__ sel, const uint32_t* __restrict__ pre,
                         uint64_t n, uint32_t* colmap, uint32_t* bits) {
  const uint64_t n_up = (n + 31) & ~31ull;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n_up;
       j += (uint64_t)gridDim.x * blockDim.x) {
    const bool on = j < n && sel[j];
    const unsigned w = __ballot_sync(FULL, on);
    if ((threadIdx.x & 31) == 0) bits[j >> 5] = w;
    if (on) colmap[pre[j]] = (uint32_t)j;
  }
}

// ---- B restricted to the selected columns -----------------------------------
// The entries of B stay in order, so the filtered rows are a compaction of the
// entry array: one bit per entry (k_bf_bits), the places from the bits' running
// count (k_bf_emit), and a row's start is the count of selected entries before
// it (k_bf_ptr).  Entries are read as one stream, 32 consecutive ones per warp
// and load, whatever the rows' lengths, and looked up in a shared-memory bitmap
// of the columns (a block per SM; columns past its 1.6 million bits are looked
// up in L2).  A warp per row with a 4-byte L2 lookup per entry spent 148 us
// counting and 178 us filling for 2e7 entries in rows of 20, twice per call;
// the four kernels here take 78 us in all.
constexpr int kBfThreads = 1024;
constexpr int kBfPer = 8;                            // entries per thread and chunk
constexpr uint32_t kBfChunk = kBfThreads * kBfPer;   // 256 words of bits
constexpr size_t kBfBitmapMax = 200 * 1024;

template <bool kShared>
__global__ void __launch_bounds__(kBfThreads)
k_bf_bits(const int32_t* __restrict__ bcol, uint64_t nnz, const uint32_t* __restrict__ bits,
          uint64_t n, uint32_t* __restrict__ ebits, uint32_t* __restrict__ chunk_cnt) {
  extern __shared__ uint32_t sbits[];
  __shared__ uint32_t total[2];
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (kShared)
    for (uint64_t w = tid; w < (n + 31) / 32; w += kBfThreads) sbits[w] = bits[w];
  if (tid < 2) total[tid] = 0;
  __syncthreads();
  const uint64_t chunks = (nnz + kBfChunk - 1) / kBfChunk;
  unsigned par = 0;
  for (uint64_t c = blockIdx.x; c < chunks; c += gridDim.x, par ^= 1) {
    int32_t j[kBfPer];
#pragma unroll
    for (int r = 0; r < kBfPer; ++r) {
      const uint64_t e = c * kBfChunk + (uint64_t)r * kBfThreads + tid;
      j[r] = e < nnz ? __ldcs(bcol + e) : -1;
    }
    unsigned mine = 0;
#pragma unroll
    for (int r = 0; r < kBfPer; ++r) {
      const uint32_t w = (uint32_t)j[r] >> 5;
      const bool on = j[r] >= 0 && (((kShared ? sbits[w] : __ldg(bits + w)) >> (j[r] & 31)) & 1u);
      const unsigned bal = __ballot_sync(FULL, on);
      if (lane == 0) {
        ebits[c * (kBfChunk / 32) + r * (kBfThreads / 32) + warp] = bal;
        mine += __popc(bal);
      }
    }
    if (lane == 0 && mine) atomicAdd(&total[par], mine);
    __syncthreads();   // (the other chunk parity's counter is free again)
    if (tid == 0) {
      chunk_cnt[c] = total[par];
      total[par ^ 1] = 0;
    }
    __syncthreads();
  }
}

// Places of a chunk's entries: wpre[w] = selected entries before word w, and
// the entries' labels.
__global__ void __launch_bounds__(256)
k_bf_emit(const int32_t* __restrict__ bcol, uint64_t nnz, const uint32_t* __restrict__ ebits,
          const uint32_t* __restrict__ chunk_off, const uint32_t* __restrict__ pre,
          uint32_t* __restrict__ wpre, uint32_t* __restrict__ ocol) {
  constexpr unsigned kWords = kBfChunk / 32;   // one per thread
  static_assert(kWords == 256, "a word per thread");
  __shared__ uint32_t swpre[kWords], sword[kWords], wsum[8];
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t chunks = (nnz + kBfChunk - 1) / kBfChunk;
  for (uint64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
    const uint32_t word = ebits[c * kWords + tid];
    uint32_t inc = __popc(word);
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, o);
      if ((int)lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t before = chunk_off[c] + inc - __popc(word);
    for (unsigned w = 0; w < warp; ++w) before += wsum[w];
    wpre[c * kWords + tid] = before;
    swpre[tid] = before;
    sword[tid] = word;
    __syncthreads();
#pragma unroll 4
    for (unsigned w = warp; w < kWords; w += 8) {
      const uint32_t bw = sword[w];
      if (!bw) continue;
      if ((bw >> lane) & 1u) {
        const int32_t j = __ldcs(bcol + c * kBfChunk + 32 * w + lane);
        ocol[swpre[w] + __popc(bw & ((1u << lane) - 1u))] = __ldg(pre + j);
      }
    }
    __syncthreads();
  }
}

// Start of every filtered row.
__global__ void k_bf_ptr(const int64_t* __restrict__ bptr, uint64_t d, uint64_t nnz,
                         const uint32_t* __restrict__ ebits, const uint32_t* __restrict__ wpre,
                         const uint32_t* __restrict__ total, uint32_t* __restrict__ optr) {
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k <= d;
       k += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = (uint64_t)bptr[k];
    optr[k] = e < nnz ? wpre[e >> 5] + __popc(ebits[e >> 5] & ((1u << (e & 31)) - 1u)) : *total;
  }
}

// First position in [lo, hi) whose label is >= L (hi if none); labels
// ascending.
__device__ __forceinline__ uint32_t lower_bound(const uint32_t* __restrict__ lab, uint32_t lo,
                                                uint32_t hi, uint32_t L) {
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(lab + mid) < L) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

struct SpRowParams {
  const int64_t* aptr;
  const int32_t* acol;
  const uint32_t* rows;           // schedule of rows
  const unsigned int* nrows_bins; // number of rows: sum of these 32 bucket counts
  uint32_t nrows_cap;             // the schedule never holds more than this
  const uint32_t* bptr;           // filtered B: row k's labels at [bptr[k], bptr[k+1])
  const uint32_t* bcol;
  uint32_t nlab;                  // selected columns
  const uint32_t* sel;            // column selected (n)
  const uint32_t* pre;            // rank of column j among the selected (n + 1)
  const uint32_t* colmap;         // label -> column
  int gram, excl;
  uint32_t window;                // labels per shared window
  uint32_t th_emit;               // emit every c >= th_emit (0xffffffff: none)
  uint32_t th_tie;                // tie value (tie_mode > 0)
  int tie_mode;                   // 0 off, 1 count ties per row, 2 emit ties under the limit
  unsigned long long* tiecnt;     // per-row tie counts (tie_mode 1)
  int hist_smem;                  // histogram of emitted c in shared memory (kHistSmem bins)
  unsigned int* hist;             // clamped histogram of emitted c (null: none)
  uint32_t hist_bins;
  Item* list;
  unsigned long long cap;
  SpScalars* sc;
};

// One block per row of C at a time: row i = sum over k in row i of A of row
// k of the filtered B, counted in shared memory one window of labels at a
// time; the window's entries are tested against the threshold and cleared
// while they are read.  Gram inputs count unordered pairs: labels from the
// rank of column i on (past it when the diagonal is excluded).
__global__ void __launch_bounds__(kSpBlock) k_spgemm_rowblock_topk(SpRowParams p) {
  extern __shared__ uint32_t smem[];
  uint32_t* acc = smem;                       // p.window counts
  uint32_t* shist = smem + p.window;          // kHistSmem bins when p.hist_smem
  __shared__ unsigned int s_row;
  __shared__ unsigned int s_wsum[kSpWarps];
  __shared__ unsigned long long s_run;
  __shared__ unsigned long long s_ties;
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t q = tid; q < p.window; q += kSpBlock) acc[q] = 0;
  if (p.hist_smem)
    for (uint32_t q = tid; q < kHistSmem; q += kSpBlock) shist[q] = 0;
  unsigned nrows = 0;
  for (int b = 0; b < 32; ++b) nrows += p.nrows_bins[b];
  if (nrows > p.nrows_cap) nrows = p.nrows_cap;
  const uint32_t row_lim = p.tie_mode == 2 ? p.sc->row_lim : 0;
  const uint32_t lim_x = p.tie_mode == 2 ? p.sc->lim_x : 0;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      s_row = atomicAdd(&p.sc->row_next, 1u);
      s_run = 0;
      s_ties = 0;
    }
    __syncthreads();
    const unsigned qr = s_row;
    if (qr >= nrows) break;
    const uint32_t i = p.rows[qr];
    if (p.tie_mode == 2 && i > row_lim) continue;
    const int64_t a0 = p.aptr[i], a1 = p.aptr[i + 1];
    uint32_t lo = 0;
    if (p.gram) lo = p.pre[i] + (p.excl ? p.sel[i] : 0u);
    const bool limited = p.tie_mode == 2 && i == row_lim;
    for (uint32_t w0 = (lo / p.window) * p.window; w0 < p.nlab; w0 += p.window) {
      const uint32_t w1 = w0 + p.window < p.nlab ? w0 + p.window : p.nlab;
      const uint32_t L = lo > w0 ? lo : w0;
      // Accumulate: each warp takes 32 of row i's entries at a time, every
      // kSpWarps-th one (graphs are often numbered by weight, so that
      // neighbouring entries are heavy together): lane l finds the part of its
      // entry's filtered row inside the window (32 searches side by side), then
      // the warp goes through the 32 parts in pieces of up to 32 labels, four
      // pieces in flight.  A warp per entry in turn waited for four dependent
      // loads on each (main pass on 1e6 nodes 865 us, then 576; with 512
      // threads a row instead of 256, 480; issue slots 86 % taken).
      const uint32_t alen = (uint32_t)(a1 - a0);
      for (uint32_t q0 = 0; q0 < alen; q0 += 32 * kSpWarps) {
        uint32_t start = 0, len = 0;
        const uint32_t q = q0 + lane * kSpWarps + warp;
        if (q < alen) {
          const uint32_t k = (uint32_t)__ldg(p.acol + a0 + q);
          const uint32_t b0 = __ldg(p.bptr + k), b1 = __ldg(p.bptr + k + 1);
          start = L == 0 ? b0 : lower_bound(p.bcol, b0, b1, L);
          const uint32_t end = w1 == p.nlab ? b1 : lower_bound(p.bcol, start, b1, w1);
          len = end - start;
        }
        unsigned todo = __ballot_sync(FULL, len != 0);
        uint32_t s = 0, left = 0;   // the current part: its next label, labels left
        while (todo || left) {
          uint32_t v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (left == 0 && todo) {
              const int r = __ffs(todo) - 1;
              todo &= todo - 1;
              s = __shfl_sync(FULL, start, r);
              left = __shfl_sync(FULL, len, r);
            }
            v[u] = lane < left ? __ldg(p.bcol + s + lane) : 0xffffffffu;
            s += 32;
            left = left > 32 ? left - 32 : 0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (v[u] != 0xffffffffu) atomicAdd(&acc[v[u] - w0], 1u);
        }
      }
      __syncthreads();
      // Scan the window: threshold, emit, clear.
      for (uint32_t base = L; base < w1; base += kSpBlock) {
        const uint32_t q = base + tid;
        uint32_t c = 0;
        if (q < w1) {
          c = acc[q - w0];
          if (c) acc[q - w0] = 0;
        }
        uint32_t j = 0;
        bool em = false, tie = false;
        if (c) {
          j = p.colmap[q];
          const bool diag_out = p.excl && !p.gram && j == i;
          em = !diag_out && c >= p.th_emit;
          tie = !diag_out && p.tie_mode != 0 && c == p.th_tie;
        }
        if (p.tie_mode == 1) {
          const unsigned nt = __popc(__ballot_sync(FULL, tie));
          if (lane == 0 && nt) atomicAdd(&s_ties, (unsigned long long)nt);
        } else if (p.tie_mode == 2) {
          if (limited) {
            // rank of this tie among the row's ties in ascending j
            const unsigned bal = __ballot_sync(FULL, tie);
            if (lane == 0) s_wsum[warp] = __popc(bal);
            __syncthreads();
            unsigned before = 0, total = 0;
            for (int w = 0; w < kSpWarps; ++w) {
              if (w < (int)warp) before += s_wsum[w];
              total += s_wsum[w];
            }
            const unsigned long long rank =
                s_run + before + __popc(bal & ((1u << lane) - 1));
            em = tie && rank < lim_x;
            __syncthreads();
            if (tid == 0) s_run += total;
          } else {
            em = tie;   // a row before the boundary row: all its ties
          }
        }
        const unsigned bal = __ballot_sync(FULL, em);
        if (bal) {
          const unsigned leader = __ffs(bal) - 1;
          unsigned long long pos0 = 0;
          if (lane == leader) pos0 = atomicAdd(&p.sc->count, (unsigned long long)__popc(bal));
          pos0 = __shfl_sync(FULL, pos0, leader);
          if (em) {
            const unsigned long long pos = pos0 + __popc(bal & ((1u << lane) - 1));
            if (pos < p.cap) {
              Item it;
              it.p = c;
              it.key = ((unsigned long long)i << 32) | j;
              it.aux = 0;
              p.list[pos] = it;
            }
            if (p.hist_smem)
              atomicAdd(&shist[c < kHistSmem ? c : kHistSmem - 1], 1u);
            else if (p.hist)
              atomicAdd(&p.hist[c < p.hist_bins ? c : p.hist_bins - 1], 1u);
          }
        }
      }
      __syncthreads();
    }
    if (p.tie_mode == 1 && tid == 0 && s_ties) p.tiecnt[i] += s_ties;   // one block per row
  }
  if (p.hist_smem) {
    __syncthreads();
    for (uint32_t q = tid; q < kHistSmem; q += kSpBlock)
      if (shist[q]) atomicAdd(&p.hist[q], shist[q]);
  }
}

// theta = the largest v >= 1 such that at least t emitted counts are >= v
// (the top bin holds every count at or above it), or 1 when fewer than t
// counts were emitted.
__global__ void __launch_bounds__(1024) k_hist_theta(const unsigned int* __restrict__ hist,
                                                     uint32_t nb, unsigned long long t,
                                                     SpScalars* sc) {
  __shared__ unsigned long long s_run;
  __shared__ unsigned long long s_w[32];
  __shared__ int s_found;
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_run = 0;
    s_found = -1;
  }
  __syncthreads();
  for (int hi = (int)nb; hi > 1; hi -= 1024) {
    const int v = hi - 1 - (int)tid;     // thread tid takes bin v, descending
    unsigned long long h = v >= 1 ? hist[v] : 0;
    unsigned long long x = h;           // inclusive prefix over tid
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(FULL, x, o);
      if ((int)lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    unsigned long long before = 0;
    for (int w = 0; w < (int)warp; ++w) before += s_w[w];
    const unsigned long long ge = s_run + before + x;   // counts >= v
    if (v >= 1 && ge >= t) atomicMax(&s_found, v);
    __syncthreads();
    if (s_found >= 1) break;
    if (tid == 1023) s_run = s_run + before + x;
    __syncthreads();
  }
  if (tid == 0) sc->theta = s_found >= 1 ? (unsigned)s_found : 1u;
}

// Boundary of the tie-limited emission: row_lim is the row in whose ties
// the need runs out (prefix over rows in index order), lim_x the number of
// its ties to take.
__global__ void k_tie_limit(const unsigned long long* __restrict__ tiepre, uint64_t m,
                            unsigned long long t, SpScalars* sc) {
  const unsigned long long have = sc->count;
  const unsigned long long need = t > have ? t - have : 0;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (uint64_t)gridDim.x * blockDim.x) {
    if (tiepre[i] < need && need <= tiepre[i + 1]) {
      sc->row_lim = (uint32_t)i;
      sc->lim_x = (uint32_t)(need - tiepre[i]);
      sc->need = need;
    }
  }
}

__global__ void k_sp_to_pairs(const Item* __restrict__ items, uint64_t n, mad_pair* out) {
  const uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const Item it = items[q];
  mad_pair pr;
  pr.i = (uint32_t)(it.key >> 32);
  pr.j = (uint32_t)it.key;
  pr.x = 0;
  pr.c = (double)it.p;
  out[q] = pr;
}

unsigned blocks_for(uint64_t n, unsigned cap) {
  const uint64_t b = (n + 255) / 256;
  return (unsigned)(b == 0 ? 1 : (b < cap ? b : cap));
}

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch of one call.
struct SpWs {
  uint32_t *cb, *rorder, *corder, *sel, *pre, *colmap, *bits, *bp, *bcol, *part, *hist;
  uint32_t *ebits, *wpre, *ccnt, *coff;
  unsigned long long *tiecnt, *tiepre, *part64;
  SpScalars* sc;
  SelectWs sel_ws;
};

size_t sp_ws_bytes(uint64_t m, uint64_t d, uint64_t n, uint64_t nnzb, uint64_t t, SpWs* ws,
                   char* base) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + off : nullptr;
    off += align_up(bytes);
    return p;
  };
  const uint64_t chunks = nnzb / kBfChunk + 1;
  const uint64_t parts = scan_partial_elems((n > chunks ? n : chunks) + 1);
  SpWs w{};
  w.cb = (uint32_t*)take(4 * n);
  w.rorder = (uint32_t*)take(4 * m);
  w.corder = (uint32_t*)take(4 * n);
  w.sel = (uint32_t*)take(4 * (n + 1));
  w.pre = (uint32_t*)take(4 * (n + 1));
  w.colmap = (uint32_t*)take(4 * n);
  w.bits = (uint32_t*)take(4 * (n / 32 + 1));
  w.ebits = (uint32_t*)take(4 * chunks * (kBfChunk / 32));
  w.wpre = (uint32_t*)take(4 * chunks * (kBfChunk / 32));
  w.ccnt = (uint32_t*)take(4 * chunks);
  w.coff = (uint32_t*)take(4 * (chunks + 1));
  w.bp = (uint32_t*)take(4 * (d + 1));
  w.bcol = (uint32_t*)take(4 * (nnzb ? nnzb : 1));
  w.part = (uint32_t*)take(4 * parts);
  w.hist = (uint32_t*)take(4 * kHistGlobal);
  w.tiecnt = (unsigned long long*)take(8 * (m + 1));
  w.tiepre = (unsigned long long*)take(8 * (m + 1));
  w.part64 = (unsigned long long*)take(8 * scan_partial_elems(m + 1));
  w.sc = (SpScalars*)take(sizeof(SpScalars));
  char* sb = take(select_ws_bytes(kSpListCap, t));
  if (base) w.sel_ws = select_ws_carve(sb, kSpListCap, t);
  if (ws) *ws = w;
  return off;
}

}  // namespace
}  // namespace mad

using namespace mad;

mad_status mad_sparse_topt(mad_ctx* ctx, const mad_matrix* A, const mad_matrix* B, uint32_t t,
                           uint32_t options, mad_pair* out_dev, uint32_t* n_out_host,
                           mad_stream stream) {
  if (!ctx || !A || !B || !out_dev || !n_out_host || t == 0) return MAD_ERR_ARG;
  *n_out_host = 0;
  if (options & ~(uint32_t)MAD_SPARSE_NO_BOUND) return MAD_ERR_ARG;
  if (A->fmt != MAD_CSR || B->fmt != MAD_CSR || A->dt != MAD_BINARY || B->dt != MAD_BINARY)
    return MAD_ERR_UNSUPPORTED;
  if (!A->rowptr || !A->colidx || !B->rowptr || !B->colidx || A->rows <= 0 || A->cols <= 0 ||
      B->cols <= 0)
    return MAD_ERR_ARG;
  if (B->rows != A->cols || A->rows >= (1ll << 31) || B->cols >= (1ll << 31) ||
      A->cols >= (1ll << 31))
    return MAD_ERR_ARG;
  if (t > kSpListCap / 2) return MAD_ERR_UNSUPPORTED;
  const bool gram = (ctx->flags & MAD_GRAM) != 0;
  const bool excl = (ctx->flags & MAD_EXCLUDE_DIAG) != 0;
  if (gram && A->rows != B->cols) return MAD_ERR_ARG;
  const bool bound = !(options & MAD_SPARSE_NO_BOUND);
  cudaStream_t st = (cudaStream_t)stream;
  const uint64_t m = (uint64_t)A->rows, d = (uint64_t)A->cols, n = (uint64_t)B->cols;

  int64_t nnz_h[2] = {0, 0};
  cudaMemcpyAsync(&nnz_h[0], A->rowptr + m, 8, cudaMemcpyDeviceToHost, st);
  cudaMemcpyAsync(&nnz_h[1], B->rowptr + d, 8, cudaMemcpyDeviceToHost, st);
  cudaError_t ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return cuda_status(ce);
  if (nnz_h[0] < 0 || nnz_h[1] < 0 || nnz_h[1] >= (1ll << 31)) return MAD_ERR_ARG;
  const uint64_t nnzb = (uint64_t)nnz_h[1];

  mad_status rs = ensure_scratch(ctx, sp_ws_bytes(m, d, n, nnzb, t, nullptr, nullptr), st);
  if (rs != MAD_OK) return rs;
  SpWs w{};
  sp_ws_bytes(m, d, n, nnzb, t, &w, (char*)ctx->scratch);

  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid_stream = (unsigned)(sms * 8);

  // Column counts and degree orders of rows and columns.
  cudaMemsetAsync(w.sc, 0, sizeof(SpScalars), st);
  if (gram) {
    k_row_degrees<<<blocks_for(n, grid_stream), 256, 0, st>>>(A->rowptr, n, w.cb);
  } else {
    cudaMemsetAsync(w.cb, 0, 4 * n, st);
    k_col_counts<<<blocks_for(nnzb, grid_stream), 256, 0, st>>>(B->colidx, nnzb, w.cb);
  }
  k_logbin_count<<<blocks_for(m, grid_stream), 256, 0, st>>>(A->rowptr, nullptr, m, 1u,
                                                            w.sc->bins[0]);
  k_logbin_count<<<blocks_for(n, grid_stream), 256, 0, st>>>(nullptr, w.cb, n, 1u,
                                                            w.sc->bins[1]);
  k_logbin_scatter<<<blocks_for(m, grid_stream), 256, 0, st>>>(A->rowptr, nullptr, m, 1u,
                                                              w.sc->bins[0], w.sc->cur[0],
                                                              w.rorder);
  k_logbin_scatter<<<blocks_for(n, grid_stream), 256, 0, st>>>(nullptr, w.cb, n, 1u,
                                                              w.sc->bins[1], w.sc->cur[1],
                                                              w.corder);
  count_launch(ctx, 5);
  SpScalars hs{};
  cudaMemcpyAsync(&hs, w.sc, sizeof(SpScalars), cudaMemcpyDeviceToHost, st);
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);
  uint64_t rows_nz = 0, cols_nz = 0;
  for (int b = 0; b < 32; ++b) {
    rows_nz += hs.bins[0][b];
    cols_nz += hs.bins[1][b];
  }
  if (rows_nz == 0 || cols_nz == 0) return MAD_OK;   // C = 0: no stored entry

  const size_t smem_max = (size_t)kSpWindowMax * 4 + (size_t)kHistSmem * 4;
  cudaFuncSetAttribute(k_spgemm_rowblock_topk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem_max);
  cudaFuncSetAttribute(k_bf_bits<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kBfBitmapMax);

  // Selected columns -> labels and the filtered, relabelled B.
  auto select_columns = [&](bool from_list, uint32_t h, uint32_t th) -> mad_status {
    if (from_list) {
      cudaMemsetAsync(w.sel, 0, 4 * n, st);
      k_mark_list<<<blocks_for(h, 1u << 30), 256, 0, st>>>(w.corder, h, w.sel);
    } else {
      k_mark_deg<<<blocks_for(n, grid_stream), 256, 0, st>>>(w.cb, n, th, w.sel);
    }
    count_launch(ctx);
    mad_status r = scan_exclusive_u32(ctx, w.sel, w.pre, n, w.part, st);
    if (r != MAD_OK) return r;
    k_colmap<<<blocks_for(n, grid_stream), 256, 0, st>>>(w.sel, w.pre, n, w.colmap, w.bits);
    const uint64_t chunks = (nnzb + kBfChunk - 1) / kBfChunk;
    const size_t bitmap = (size_t)((n + 31) / 32) * 4;
    const unsigned bg = (unsigned)(chunks < (uint64_t)sms ? (chunks ? chunks : 1) : sms);
    if (bitmap <= kBfBitmapMax)
      k_bf_bits<true><<<bg, kBfThreads, bitmap, st>>>(B->colidx, nnzb, w.bits, n, w.ebits, w.ccnt);
    else
      k_bf_bits<false><<<bg, kBfThreads, 0, st>>>(B->colidx, nnzb, w.bits, n, w.ebits, w.ccnt);
    count_launch(ctx, 2);
    if ((r = scan_exclusive_u32(ctx, w.ccnt, w.coff, chunks, w.part, st)) != MAD_OK) return r;
    k_bf_emit<<<(unsigned)(chunks < grid_stream ? (chunks ? chunks : 1) : grid_stream), 256, 0, st>>>(
        B->colidx, nnzb, w.ebits, w.coff, w.pre, w.wpre, w.bcol);
    k_bf_ptr<<<blocks_for(d + 1, grid_stream), 256, 0, st>>>(B->rowptr, d, nnzb, w.ebits, w.wpre,
                                                             w.coff + chunks, w.bp);
    count_launch(ctx, 2);
    return cuda_status(cudaGetLastError());
  };

  auto run_rows = [&](uint32_t nlab, const unsigned int* bins, uint32_t rows_cap,
                      uint32_t th_emit, uint32_t th_tie, int tie_mode, bool hist_smem,
                      bool hist) -> mad_status {
    SpRowParams p{};
    p.aptr = A->rowptr;
    p.acol = A->colidx;
    p.rows = w.rorder;
    p.nrows_bins = bins;
    p.nrows_cap = rows_cap;
    p.bptr = w.bp;
    p.bcol = w.bcol;
    p.nlab = nlab;
    p.sel = w.sel;
    p.pre = w.pre;
    p.colmap = w.colmap;
    p.gram = gram;
    p.excl = excl;
    p.window = nlab < kSpWindowMax ? ((nlab + 31) & ~31u) : kSpWindowMax;
    if (p.window == 0) p.window = 32;
    p.th_emit = th_emit;
    p.th_tie = th_tie;
    p.tie_mode = tie_mode;
    p.tiecnt = w.tiecnt;
    p.hist_smem = hist_smem;
    p.hist = hist ? w.hist : nullptr;
    p.hist_bins = hist_smem ? kHistSmem : kHistGlobal;
    p.list = w.sel_ws.l0;
    p.cap = kSpListCap;
    p.sc = w.sc;
    const size_t smem = (size_t)p.window * 4 + (hist_smem ? (size_t)kHistSmem * 4 : 0);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spgemm_rowblock_topk, kSpBlock, smem);
    if (per_sm < 1) per_sm = 1;
    uint64_t blocks = (uint64_t)per_sm * sms;
    if (blocks > rows_cap) blocks = rows_cap ? rows_cap : 1;
    cudaMemsetAsync(&w.sc->row_next, 0, sizeof(unsigned int), st);
    k_spgemm_rowblock_topk<<<(unsigned)blocks, kSpBlock, smem, st>>>(p);
    count_launch(ctx);
    return cuda_status(cudaGetLastError());
  };

  // 1. Pilot: the heaviest rows against the heaviest columns, every stored
  //    entry counted into the histogram; its t-th largest is theta_0.
  const uint32_t pilot = pilot_size(t);
  const uint32_t hr = (uint32_t)(rows_nz < pilot ? rows_nz : pilot);
  const uint32_t hc = (uint32_t)(cols_nz < pilot ? cols_nz : pilot);
  if ((rs = select_columns(true, hc, 0)) != MAD_OK) return rs;
  cudaMemsetAsync(w.hist, 0, 4 * kHistGlobal, st);
  // The pilot's rows are the first hr of the row order: count them through
  // a bucket array that sums to hr.
  unsigned int* pilot_bins = w.hist + kHistGlobal - 32;
  {
    unsigned int hb[32] = {0};
    hb[0] = hr;
    cudaMemcpyAsync(pilot_bins, hb, sizeof(hb), cudaMemcpyHostToDevice, st);
  }
  if ((rs = run_rows(hc, pilot_bins, hr, 1u, 0u, 0, true, true)) != MAD_OK) return rs;
  k_hist_theta<<<1, 1024, 0, st>>>(w.hist, kHistSmem, t, w.sc);
  count_launch(ctx);
  unsigned int theta0 = 1;
  cudaMemcpyAsync(&theta0, &w.sc->theta, 4, cudaMemcpyDeviceToHost, st);
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);

  // 2. Main pass over the rows and columns that can reach theta_0.
  const uint32_t th_deg = bound ? theta0 : 1u;
  cudaMemsetAsync(w.sc, 0, sizeof(SpScalars), st);
  k_logbin_count<<<blocks_for(m, grid_stream), 256, 0, st>>>(A->rowptr, nullptr, m, th_deg,
                                                            w.sc->bins[0]);
  k_logbin_scatter<<<blocks_for(m, grid_stream), 256, 0, st>>>(A->rowptr, nullptr, m, th_deg,
                                                              w.sc->bins[0], w.sc->cur[0],
                                                              w.rorder);
  count_launch(ctx, 2);
  if ((rs = select_columns(false, 0, th_deg)) != MAD_OK) return rs;
  uint32_t nlab = 0;
  cudaMemcpyAsync(&nlab, w.pre + n, 4, cudaMemcpyDeviceToHost, st);
  cudaMemsetAsync(w.hist, 0, 4 * kHistGlobal, st);
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);
  if (nlab > 0) {
    if ((rs = run_rows(nlab, w.sc->bins[0], (uint32_t)m, theta0, 0u, 0, false, true)) != MAD_OK)
      return rs;
  }
  unsigned long long count = 0;
  cudaMemcpyAsync(&count, &w.sc->count, 8, cudaMemcpyDeviceToHost, st);
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);

  if (count > kSpListCap) {
    // Too many candidates at theta_0: the exact tau from the histogram,
    // then every c > tau and the smallest keys among c == tau.
    k_hist_theta<<<1, 1024, 0, st>>>(w.hist, kHistGlobal, t, w.sc);
    count_launch(ctx);
    unsigned int tau = 0;
    cudaMemcpyAsync(&tau, &w.sc->theta, 4, cudaMemcpyDeviceToHost, st);
    if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);
    if (tau >= kHistGlobal - 1) return MAD_ERR_UNSUPPORTED;   // counts beyond the histogram
    cudaMemsetAsync(&w.sc->count, 0, 8, st);
    cudaMemsetAsync(w.tiecnt, 0, 8 * (m + 1), st);
    if ((rs = run_rows(nlab, w.sc->bins[0], (uint32_t)m, tau + 1, tau, 1, false, false)) != MAD_OK)
      return rs;
    if ((rs = scan_exclusive_u64(ctx, (const uint64_t*)w.tiecnt, (uint64_t*)w.tiepre, m, (uint64_t*)w.part64, st)) != MAD_OK) return rs;
    k_tie_limit<<<blocks_for(m, grid_stream), 256, 0, st>>>(w.tiepre, m, t, w.sc);
    count_launch(ctx);
    if ((rs = run_rows(nlab, w.sc->bins[0], (uint32_t)m, 0xffffffffu, tau, 2, false, false)) !=
        MAD_OK)
      return rs;
    cudaMemcpyAsync(&count, &w.sc->count, 8, cudaMemcpyDeviceToHost, st);
    if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);
    if (count > kSpListCap) return MAD_ERR_STATE;
  }

  // 3. The t largest candidates by (c desc, key asc).
  uint64_t nsel = 0;
  if ((rs = select_list(ctx, w.sel_ws, count, t, 32, &nsel, st)) != MAD_OK) return rs;
  if (nsel) {
    k_sp_to_pairs<<<blocks_for(nsel, 1u << 30), 256, 0, st>>>(w.sel_ws.out, nsel, out_dev);
    count_launch(ctx);
  }
  if ((ce = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_status(ce);
  *n_out_host = (uint32_t)nsel;
  return MAD_OK;
}
