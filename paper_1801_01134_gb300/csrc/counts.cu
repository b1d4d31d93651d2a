// N_blocks(r,c) of all twelve shapes from a CSR, without conversion (section
// "Performance polynomial interpolation": the selection inputs Avg(r,c) =
// nnz / N_blocks(r,c) are cheap to compute) plus the row-length statistics of
// the selection features, all in one pass over the column indices.
//
// A thread block takes 128 consecutive rows (sixteen 8-row groups) at a time
// and works through them in steps of whole groups that hold at most kCap
// entries, in shared memory. The sorted columns of the rows are the lists of
// r = 1; merging neighbouring lists two by two gives the interval lists of
// r = 2, 4 and 8. The merged places are dealt out evenly, a few consecutive
// ones per thread: a thread finds by halving how many of the places before
// its own come from each list (the merge path) and goes on from there entry
// by entry, so rows of any length fill the threads alike.
// The greedy cover of a list splits at every gap of at least c: the block
// holding the left column ends before the right one. So the runs between gaps
// of 16 are covered independently for c = 4, 8 and 16. A run of one entry is
// one block and is counted in passing; longer runs go to a queue and are
// walked block by block, one thread per run and c.
// Groups with more than kCap entries (power-law hubs) are cut along their
// longest row into column ranges at columns that start a block in every cover
// (no column of the group in the 16 before them; k_count_cuts), one thread
// block per range (k_count_long); a range that still holds more than a step's
// entries is taken in steps that hand on where each list's last blocks start.
//
// What bounds it: instructions (about a dozen per entry and merge, in shared
// memory); DRAM reads are the column indices once. Before, the counts of
// r = 1 searched every entry's row in the whole row pointer and one thread
// merged all rows of an interval of up to 1024 entries, once for each r, with
// the host in between: R-MAT scale 20, 15.7 M entries, 3.4 ms of
// kernels, now 0.40 (spc5_select with the network 4.31 -> 0.48 ms). (Merging by one search per entry took
// 0.62 ms, and 1.0 ms without the repeated columns, which takes a prefix sum
// per merge.)
// All counts are integers summed with atomics, so the order of the sums does
// not matter.
#include <climits>

#include "internal.cuh"

namespace spc5 {
namespace {

constexpr int kCntThreads = 256;
constexpr int kCap = 9 * kCntThreads;  // entries of one step: nine places per thread (odd: no bank conflicts)
constexpr int kCntRows = 128;          // rows a thread block takes at a time
constexpr int kLists = 15;             // lists of one 8-row group: 8 + 4 + 2 + 1
constexpr int kPiece = 1536;           // entries of a long group's column range, about
constexpr int kCandidates = 256;       // entries looked at for a range's start
// queued runs hold at least two of a level's entries, so a thread's nine places
// give at most five; a carried step queues the first and last run of each list
// too, and a list's last entry is queued by itself where it lies within 16 of
// INT_MAX, which stands behind every list
constexpr int kQueue = 4 * 5 * kCntThreads + kLists * (kCntRows / 8) + 2 * kLists + 2;
constexpr int kCntPerSm = 4;           // thread blocks per SM of the persistent grid (50 KB of shared memory each)

struct CountShared {
  int32_t col[4][kCap];        // the lists of r = 1, 2, 4, 8, each where its first row's entries start
  uint16_t queue[kQueue];      // runs to walk: level * kCap + place of the first column
  uint8_t row[kCap];           // row of a place, counted from the step's first
  int32_t rel[kCntRows + 1];   // row starts of the thread block's rows
  int32_t off[kCntRows + 1];   // row starts of the step's rows
  int32_t open[2][kLists][3];  // carried steps: first columns of the open blocks, before and after the step
  int nqueue;
  int32_t cut;                 // smallest column found
  unsigned long long sum[12];
  int64_t cur[8], end[8];      // k_count_long: the rows' entries still to take
};

struct CountTask {  // one column range of a long group
  int64_t group;      // < 0: no range (see list_ranges)
  int32_t row, piece;  // its longest row, number of the range
};

struct CountCut {  // where the range starts: the first column, or INT_MAX, and each row's first entry
  int64_t at[8];
  int32_t column;
};

// ranges of a long group of `total` entries
__host__ __device__ __forceinline__ int64_t pieces_of(int64_t total) { return (total + kPiece - 1) / kPiece; }

// Column b starts a new run after a: they lie at least 16 apart. Unsigned, so
// that the whole range [-16, 2^31) works (-16 stands before a list's first
// column).
__device__ __forceinline__ bool apart(int32_t a, int32_t b) { return (uint32_t)b - (uint32_t)a >= 16u; }

// Lists the `np` ranges of a long group, by one warp. The list has room for
// `cap`, which is enough for row pointers that ascend from 0 to nnz; the caller
// may not have checked them, and pointers that fall back between two thread
// blocks' rows hold more. A group whose ranges do not all fit is left out.
__device__ __forceinline__ void list_ranges(CountTask* __restrict__ tasks, unsigned long long* __restrict__ ntasks,
                                            int64_t cap, int64_t group, int longest, int64_t np) {
  const int lane = threadIdx.x & 31;
  unsigned long long first = 0;
  if (lane == 0) first = atomicAdd(ntasks, (unsigned long long)np);
  const int64_t at = (int64_t)__shfl_sync(0xffffffffu, first, 0);
  const bool fits = at + np <= cap;
  for (int64_t j = lane; j < np && at + j < cap; j += 32)
    tasks[at + j] = CountTask{fits ? group : -1, longest, (int)j};
}

// the ranges that were listed
__device__ __forceinline__ int64_t listed_ranges(const unsigned long long* __restrict__ ntasks, int64_t cap) {
  const unsigned long long nt = *ntasks;
  return nt < (unsigned long long)cap ? (int64_t)nt : cap;
}

// lists before level k's in CountShared::open
__device__ __forceinline__ int open_base(int k) { return 16 - (16 >> k); }

// the runs at places d0 + i (bit i of `runs`) of level k into the queue; all
// lanes of the warp call it
__device__ __forceinline__ void queue_runs(CountShared& sh, uint32_t runs, int k, int d0) {
  if (!__any_sync(0xffffffffu, runs != 0u)) return;
  const int lane = threadIdx.x & 31;
  const int mine = __popc(runs);
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  int at = 0;
  if (lane == 31) at = atomicAdd(&sh.nqueue, incl);
  at = __shfl_sync(0xffffffffu, at, 31) + incl - mine;
  for (; runs; runs &= runs - 1) sh.queue[at++] = (uint16_t)(k * kCap + d0 + __ffs(runs) - 1);
}

// Level 0: the rows themselves. Fills sh.row; runs of one entry are counted
// (the result), longer ones queued. With CARRY the first run of a list may
// continue an earlier block and the last one may run on, so both are queued
// whatever their length.
template <bool CARRY>
__device__ __forceinline__ unsigned row_runs(CountShared& sh, int rows, int total, int per) {
  const int d0 = threadIdx.x * per, d1 = min(d0 + per, total);
  unsigned single = 0;
  uint32_t runs = 0u;
  if (d0 < d1) {
    int r = 0, b = rows;  // last row starting at or before d0
    while (b - r > 1) {
      const int mid = (r + b) >> 1;
      if (sh.off[mid] <= d0) r = mid; else b = mid;
    }
    int base = sh.off[r], end = sh.off[r + 1];
    int32_t prev = d0 > base ? sh.col[0][d0 - 1] : -16;
    int32_t c = sh.col[0][d0];
    for (int d = d0; d < d1; ++d) {
      while (d >= end) {
        ++r;
        base = end;
        end = sh.off[r + 1];
      }
      if (d == base) prev = -16;
      sh.row[d] = (uint8_t)r;
      const int32_t after = d + 1 < total ? sh.col[0][d + 1] : INT_MAX;
      const int32_t next = d + 1 < end ? after : INT_MAX;
      if (apart(prev, c)) {
        if (!apart(c, next) || (CARRY && (d == base || d + 1 == end)))
          runs |= 1u << (d - d0);
        else
          ++single;
      }
      prev = c;
      c = after;
    }
  }
  queue_runs(sh, runs, 0, d0);
  __syncthreads();
  return single;
}

// Lists of level k (2^k rows each) from those of level k - 1, and their runs
// as in row_runs.
template <bool CARRY>
__device__ __forceinline__ unsigned merge_lists(CountShared& sh, int k, int total, int per) {
  const int32_t* __restrict__ src = sh.col[k - 1];
  int32_t* __restrict__ dst = sh.col[k];
  const int d0 = threadIdx.x * per, d1 = min(d0 + per, total);
  unsigned single = 0;
  uint32_t runs = 0u;
  if (d0 < d1) {
    const int half = 1 << (k - 1);
    int p = (sh.row[d0] >> k) << k;  // the list's first row
    int base = sh.off[p], mid = sh.off[p + half], end = sh.off[p + 2 * half];
    // entries of the first list among the diag places before d0
    const int diag = d0 - base;
    int lo = max(0, diag - (end - mid)), hi = min(diag, mid - base);
    while (lo < hi) {
      const int m = (lo + hi) >> 1;
      if (src[base + m] <= src[mid + diag - 1 - m]) lo = m + 1; else hi = m;
    }
    int i = base + lo, j = mid + diag - lo;
    int32_t prev = -16;
    if (i > base) prev = src[i - 1];
    if (j > mid) prev = max(prev, src[j - 1]);
    int32_t x = i < mid ? src[i] : INT_MAX, y = j < end ? src[j] : INT_MAX;
    for (int d = d0; d < d1; ++d) {
      if (d >= end) {  // the next list that holds entries
        p = (sh.row[d] >> k) << k;
        base = d;
        mid = sh.off[p + half];
        end = sh.off[p + 2 * half];
        i = base;
        j = mid;
        x = i < mid ? src[i] : INT_MAX;
        y = j < end ? src[j] : INT_MAX;
        prev = -16;
      }
      const int32_t c = min(x, y);
      if (x <= y) {
        ++i;
        x = i < mid ? src[i] : INT_MAX;
      } else {
        ++j;
        y = j < end ? src[j] : INT_MAX;
      }
      dst[d] = c;
      if (apart(prev, c)) {
        if (!apart(c, min(x, y)) || (CARRY && (d == base || d + 1 == end)))
          runs |= 1u << (d - d0);
        else
          ++single;
      }
      prev = c;
    }
  }
  queue_runs(sh, runs, k, d0);
  __syncthreads();
  return single;
}

// first place of [i, stop) whose column lies at least C after `first`
// (doubling steps, then halving: blocks end a few places on)
template <int C>
__device__ __forceinline__ int block_end(const int32_t* __restrict__ col, int i, int stop, int32_t first) {
  int lo = i, step = 1;
  while (i < stop && (uint32_t)col[i] - (uint32_t)first < (uint32_t)C) {
    lo = i + 1;
    i += step;
    step <<= 1;
  }
  int hi = i < stop ? i : stop;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if ((uint32_t)col[mid] - (uint32_t)first < (uint32_t)C) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// the queued runs' blocks for one c (the q-th), added to cnt[level][q]
template <bool CARRY, int Q>
__device__ __forceinline__ void walk_runs(CountShared& sh, unsigned (&cnt)[4][3]) {
  constexpr int C = 4 << Q;
  unsigned long long found = 0;  // 16 bits per level: a step has fewer blocks
  const int nq = sh.nqueue;
#pragma unroll 1
  for (int e = threadIdx.x; e < nq; e += kCntThreads) {
    const int k = sh.queue[e] / kCap, s = sh.queue[e] % kCap;
    const int l = sh.row[s] >> k;
    const int stop = sh.off[(l + 1) << k];
    const int32_t* __restrict__ col = sh.col[k];
    int i = s;
    if (CARRY && s == sh.off[l << k]) {
      i = block_end<C>(col, s, stop, sh.open[0][open_base(k) + l][Q]);  // past the open block
      if (i == stop || (i > s && apart(col[i - 1], col[i]))) continue;
    }
    unsigned n = 0;
    for (;;) {
      ++n;
      const int32_t first = col[i];
      i = block_end<C>(col, i + 1, stop, first);
      if (i == stop) {
        if (CARRY) sh.open[1][open_base(k) + l][Q] = first;
        break;
      }
      if (apart(col[i - 1], col[i])) break;  // the next run
    }
    found += (unsigned long long)n << (16 * k);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) cnt[k][Q] += (unsigned)(found >> (16 * k)) & 0xffffu;
}

// The lists of whole 8-row groups (sh.off and sh.col[0] filled, `rows` rows,
// `total` entries) counted into cnt[level][c]. Every thread of the block
// calls it.
template <bool CARRY>
__device__ __forceinline__ void count_lists(CountShared& sh, int rows, int total, unsigned (&cnt)[4][3]) {
  if (threadIdx.x == 0) sh.nqueue = 0;
  if (CARRY && threadIdx.x < kLists * 3)
    sh.open[1][threadIdx.x / 3][threadIdx.x % 3] = sh.open[0][threadIdx.x / 3][threadIdx.x % 3];
  __syncthreads();
  const int per = ((total + kCntThreads - 1) / kCntThreads) | 1;  // places per thread
  const unsigned single = row_runs<CARRY>(sh, rows, total, per);
#pragma unroll
  for (int q = 0; q < 3; ++q) cnt[0][q] += single;
#pragma unroll 1
  for (int k = 1; k < 4; ++k) {
    const unsigned more = merge_lists<CARRY>(sh, k, total, per);
#pragma unroll
    for (int j = 1; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 3; ++q) cnt[j][q] += k == j ? more : 0u;
  }
  walk_runs<CARRY, 0>(sh, cnt);
  walk_runs<CARRY, 1>(sh, cnt);
  walk_runs<CARRY, 2>(sh, cnt);
  __syncthreads();  // the lists and the queue are free again
  if (CARRY && threadIdx.x < kLists * 3)
    sh.open[0][threadIdx.x / 3][threadIdx.x % 3] = sh.open[1][threadIdx.x / 3][threadIdx.x % 3];
}

// the block's counts into acc (one atomic per count and thread block)
__device__ __forceinline__ void add_counts(CountShared& sh, const unsigned (&cnt)[4][3],
                                           unsigned long long* __restrict__ acc) {
  if (threadIdx.x < 12) sh.sum[threadIdx.x] = 0ull;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const unsigned v = __reduce_add_sync(0xffffffffu, cnt[k][q]);
      if ((threadIdx.x & 31) == 0 && v) atomicAdd(&sh.sum[3 * k + q], (unsigned long long)v);
    }
  __syncthreads();
  if (threadIdx.x < 12 && sh.sum[threadIdx.x]) atomicAdd(&acc[threadIdx.x], sh.sum[threadIdx.x]);
}

// Persistent blocks over the 128-row pieces of the matrix: the groups of at
// most kCap entries counted, longer ones listed as tasks. acc[13] += squared
// row lengths, acc[14] = longest row (acc[12], their sum, is nnz).
// Rows whose pointers run backwards or leave [0, nnz] are passed over (with
// their neighbours): the caller may not have checked the CSR, and on one that is
// not valid the three kernels stay inside their arrays and count something.
__global__ void __launch_bounds__(kCntThreads, kCntPerSm) k_count(int64_t n, int64_t nnz,
                                                                  const int64_t* __restrict__ rowptr,
                                                                  const int32_t* __restrict__ colidx,
                                                                  unsigned long long* __restrict__ acc,
                                                                  CountTask* __restrict__ tasks,
                                                                  unsigned long long* __restrict__ ntasks,
                                                                  int64_t cap) {
  extern __shared__ __align__(16) unsigned char raw[];
  CountShared& sh = *reinterpret_cast<CountShared*>(raw);
  unsigned cnt[4][3] = {};
  unsigned long long squares = 0, longest = 0;
  const int64_t pieces = (n + kCntRows - 1) / kCntRows;
  for (int64_t t = blockIdx.x; t < pieces; t += gridDim.x) {
    const int64_t row0 = t * kCntRows;
    const int64_t base = rowptr[row0];
    bool bad = false;
    if (threadIdx.x <= kCntRows) {
      const int64_t at = row0 + threadIdx.x < n ? row0 + threadIdx.x : n;
      const int64_t a = rowptr[at], before = at > row0 ? rowptr[at - 1] : a;
      sh.rel[threadIdx.x] = (int32_t)(a - base);
      bad = before < 0 || a < before || a > nnz;
    }
    if (__syncthreads_or(bad)) continue;  // whole block
    if (threadIdx.x < kCntRows) {
      const unsigned long long len = (unsigned long long)(sh.rel[threadIdx.x + 1] - sh.rel[threadIdx.x]);
      squares += len * len;
      longest = len > longest ? len : longest;
    }
    int g0 = 0;
    while (g0 < kCntRows / 8) {  // the same walk in every thread
      const int32_t start = sh.rel[8 * g0];
      const int32_t own = sh.rel[8 * g0 + 8] - start;
      if (own > kCap) {
        int best = 0, most = 0;
        for (int i = 0; i < 8; ++i) {
          const int32_t len = sh.rel[8 * g0 + i + 1] - sh.rel[8 * g0 + i];
          if (len > most) {
            most = len;
            best = i;
          }
        }
        if (threadIdx.x < 32) list_ranges(tasks, ntasks, cap, row0 / 8 + g0, best, pieces_of(own));
        ++g0;
        continue;
      }
      int g1 = g0 + 1;
      while (g1 < kCntRows / 8 && sh.rel[8 * g1 + 8] - start <= kCap) ++g1;
      const int rows = 8 * (g1 - g0), total = sh.rel[8 * g1] - start;
      if (total > 0) {
        for (int r = threadIdx.x; r <= rows; r += kCntThreads) sh.off[r] = sh.rel[8 * g0 + r] - start;
#pragma unroll 3
        for (int s = threadIdx.x; s < total; s += kCntThreads) sh.col[0][s] = __ldg(colidx + base + start + s);
        count_lists<false>(sh, rows, total, cnt);
      }
      g0 = g1;
    }
    __syncthreads();  // rel is free again
  }
  add_counts(sh, cnt, acc);
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    squares += __shfl_xor_sync(0xffffffffu, squares, d);
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, longest, d);
    longest = o > longest ? o : longest;
  }
  if ((threadIdx.x & 31) == 0 && longest) {
    atomicAdd(&acc[13], squares);
    atomicMax(&acc[14], longest);
  }
}

// first entry of [a, e) with a column of at least c
__device__ __forceinline__ int64_t entry_from(const int32_t* __restrict__ colidx, int64_t a, int64_t e, int32_t c) {
  while (a < e) {
    const int64_t mid = (a + e) >> 1;
    if (colidx[mid] < c) a = mid + 1; else e = mid;
  }
  return a;
}

// The start of each task's range, a warp per task: the first clean column -
// none of the group's columns in the 16 before it - among the longest row's
// entries from the range's share of it on, 32 candidates at a time; none
// among kCandidates: the range before runs on. The rows' entries around the
// candidates are bracketed first, so that these search a few hundred entries
// that the L1 holds.
__global__ void __launch_bounds__(kCntThreads) k_count_cuts(int64_t n, const int64_t* __restrict__ rowptr,
                                                            const int32_t* __restrict__ colidx,
                                                            const CountTask* __restrict__ tasks,
                                                            const unsigned long long* __restrict__ ntasks, int64_t cap,
                                                            CountCut* __restrict__ cuts) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t nt = listed_ranges(ntasks, cap);
  for (int64_t t = ((int64_t)blockIdx.x * kCntThreads + threadIdx.x) >> 5; t < nt;
       t += (int64_t)gridDim.x * (kCntThreads / 32)) {
    const CountTask tk = tasks[t];
    if (tk.group < 0) continue;  // whole warp
    const int64_t row0 = tk.group * 8;
    const int64_t first = rowptr[row0 + tk.row], len = rowptr[row0 + tk.row + 1] - first;
    const int64_t np = pieces_of(rowptr[row0 + 8 < n ? row0 + 8 : n] - rowptr[row0]);
    const int64_t share = (len + np - 1) / np;  // entries of the longest row per range
    const int64_t p0 = tk.piece * share;
    const int64_t few = share < kCandidates ? share : kCandidates;
    const int64_t p1 = p0 + few < len ? p0 + few : len;
    if (p0 >= p1) {  // whole warp
      if (lane == 0) cuts[t].column = INT_MAX;
      continue;
    }
    // lanes 0-7: each row's first entry that the candidates may look at, lanes 8-15: the end
    int64_t mine = 0;
    if (lane < 16) {
      const int i = lane & 7;
      const int64_t a = row0 + i < n ? rowptr[row0 + i] : 0, e = row0 + i < n ? rowptr[row0 + i + 1] : 0;
      mine = lane < 8 ? entry_from(colidx, a, e, colidx[first + p0] - 16) : entry_from(colidx, a, e, colidx[first + p1 - 1]);
    }
    int32_t cut = INT_MAX;
    for (int64_t p = p0; p < p1 && cut == INT_MAX; p += 32) {
      bool clean = p + lane < p1;
      const int32_t c = clean ? colidx[first + p + lane] : INT_MAX;
      for (int i = 0; i < 8; ++i) {
        const int64_t a = __shfl_sync(kAll, mine, i), e = __shfl_sync(kAll, mine, i + 8);
        if (clean) {
          const int64_t q = entry_from(colidx, a, e, c);  // c is at most the last candidate
          clean = !(q > a && colidx[q - 1] > c - 16);
        }
      }
      const unsigned who = __ballot_sync(kAll, clean);
      if (who) cut = __shfl_sync(kAll, c, __ffs(who) - 1);
    }
    const int64_t e = __shfl_sync(kAll, mine, (lane & 7) + 8);
    if (lane < 8 && cut != INT_MAX) cuts[t].at[lane] = entry_from(colidx, mine, e, cut);
    if (lane == 0) cuts[t].column = cut;
  }
}

__global__ void __launch_bounds__(kCntThreads, kCntPerSm) k_count_long(int64_t n, const int64_t* __restrict__ rowptr,
                                                                       const int32_t* __restrict__ colidx,
                                                                       const CountTask* __restrict__ tasks,
                                                                       const CountCut* __restrict__ cuts,
                                                                       const unsigned long long* __restrict__ ntasks,
                                                                       int64_t cap, unsigned long long* __restrict__ acc) {
  extern __shared__ __align__(16) unsigned char raw[];
  CountShared& sh = *reinterpret_cast<CountShared*>(raw);
  unsigned cnt[4][3] = {};
  const int64_t nt = listed_ranges(ntasks, cap);
  for (int64_t t = blockIdx.x; t < nt; t += gridDim.x) {
    const CountTask tk = tasks[t];
    if (tk.group < 0) continue;  // whole block
    if (tk.piece > 0 && cuts[t].column == INT_MAX) continue;  // the range before runs on through this one
    const int64_t row0 = tk.group * 8;
    // the group's tasks follow one another
    const int64_t after = t - tk.piece + pieces_of(rowptr[row0 + 8 < n ? row0 + 8 : n] - rowptr[row0]);
    int64_t next = t + 1;
    while (next < after && cuts[next].column == INT_MAX) ++next;
    if (threadIdx.x < 8) {
      const int64_t r = row0 + threadIdx.x;
      const int64_t a = r < n ? rowptr[r] : 0, e = r < n ? rowptr[r + 1] : 0;
      // both lie in the row; columns out of order can put the end before the
      // start, and one row's negative share would hide another's length below
      const int64_t from = tk.piece > 0 ? cuts[t].at[threadIdx.x] : a;
      const int64_t to = next < after ? cuts[next].at[threadIdx.x] : e;
      sh.cur[threadIdx.x] = from;
      sh.end[threadIdx.x] = to > from ? to : from;
    }
    if (threadIdx.x < kLists * 3) sh.open[0][threadIdx.x / 3][threadIdx.x % 3] = -16;
    for (;;) {
      // all that is left where it fits a step; else up to an eighth of a step
      // of each row, cut where the first row that has more goes on, so that a
      // column's entries come in the same step
      __syncthreads();
      if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int64_t a = 0, e = 0;
        if (lane < 8) {
          a = sh.cur[lane];
          e = sh.end[lane];
        }
        int64_t left = e - a;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) left += __shfl_xor_sync(0xffffffffu, left, d);
        if (left > kCap) {  // whole warp
          int32_t cut = INT_MAX;
          if (e - a > kCap / 8) {
            e = a + kCap / 8;
            cut = colidx[e];
          }
          cut = __reduce_min_sync(0xffffffffu, cut);
          if (lane < 8) e = entry_from(colidx, a, e, cut);
        }
        const int take = (int)(e - a);
        int incl = take;
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += v;
        }
        if (lane < 8) sh.off[lane + 1] = incl;
        if (lane == 0) sh.off[0] = 0;
      }
      __syncthreads();
      const int total = sh.off[8];
      if (total == 0) break;  // whole block
      {
        const int i = threadIdx.x >> 5;  // a warp per row
        const int32_t* __restrict__ from = colidx + sh.cur[i] - sh.off[i];
        for (int s = sh.off[i] + (threadIdx.x & 31); s < sh.off[i + 1]; s += 32) sh.col[0][s] = __ldg(from + s);
      }
      __syncthreads();
      if (threadIdx.x < 8) sh.cur[threadIdx.x] += sh.off[threadIdx.x + 1] - sh.off[threadIdx.x];
      count_lists<true>(sh, 8, total, cnt);
    }
  }
  add_counts(sh, cnt, acc);
}

}  // namespace

// acc (device, 15 entries, zeroed here): [0..11] N_blocks in the order r in
// {1,2,4,8} outer, c in {4,8,16} inner; [12..14] sum, sum of squares and max of
// the row lengths.
cudaError_t launch_block_counts(int64_t n, int64_t nnz, const int64_t* rowptr, const int32_t* colidx,
                                unsigned long long* acc, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 15, s);
  if (e != cudaSuccess || n <= 0) return e;
  // a long group of L > kCap entries has at most L / kPiece + 1 ranges; a
  // group is long only where the matrix has more than kCap entries
  const int64_t cap = nnz > kCap ? nnz / kPiece + nnz / kCap + 1 : 1;
  struct Scratch {  // ntasks, then the tasks and their cuts
    void* p = nullptr;
    cudaStream_t s;
    ~Scratch() {
      if (p) cudaFreeAsync(p, s);
    }
  } buf{nullptr, s};
  e = pool_alloc(&buf.p, 16 + (sizeof(CountTask) + sizeof(CountCut)) * (size_t)cap, s);
  if (e != cudaSuccess) return e;
  unsigned long long* ntasks = (unsigned long long*)buf.p;
  CountTask* tasks = (CountTask*)(ntasks + 2);
  CountCut* cuts = (CountCut*)(tasks + cap);
  e = cudaMemsetAsync(ntasks, 0, sizeof(unsigned long long), s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(acc + 12, rowptr + n, sizeof(int64_t), cudaMemcpyDeviceToDevice, s);  // the row lengths' sum
  const int smem = (int)sizeof(CountShared);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_count, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_count_long, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int64_t pieces = (n + kCntRows - 1) / kCntRows;
  const int64_t most = (int64_t)sm_count() * kCntPerSm;
  k_count<<<(unsigned)(pieces < most ? pieces : most), kCntThreads, smem, s>>>(n, nnz, rowptr, colidx, acc, tasks,
                                                                                ntasks, cap);
  if (nnz > kCap) {
    const int64_t cut_blocks = (int64_t)sm_count() * 8, want = (cap * 32 + kCntThreads - 1) / kCntThreads;
    k_count_cuts<<<(unsigned)(want < cut_blocks ? want : cut_blocks), kCntThreads, 0, s>>>(n, rowptr, colidx, tasks,
                                                                                         ntasks, cap, cuts);
    k_count_long<<<(unsigned)(cap < most ? cap : most), kCntThreads, smem, s>>>(n, rowptr, colidx, tasks, cuts, ntasks,
                                                                                cap, acc);
  }
  return cudaGetLastError();
}

spc5_status count_blocks_impl(int64_t n, int64_t nnz, const int64_t* rowptr, const int32_t* colidx,
                              int64_t* nblocks_out, cudaStream_t s) {
  unsigned long long* acc = nullptr;
  cudaError_t e = pool_alloc((void**)&acc, sizeof(unsigned long long) * 16, s);
  if (e != cudaSuccess) return cuda_fail(e, "count_blocks: scratch");
  unsigned long long h[15];
  e = launch_block_counts(n, nnz, rowptr, colidx, acc, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(acc, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "count_blocks");
  for (int q = 0; q < 12; ++q) nblocks_out[q] = (int64_t)h[q];
  return SPC5_OK;
}

}  // namespace spc5
