// fcs_sort.cu - deterministic mode: group the (cell, task, count) records of
// the hit kernel by cell and fold each cell in ascending task order:
//   E_cell = fold_{tasks ascending} fl32( fl32(n_cell,task) * Ehit_task )
// starting from 0.0f.  Every hit of a task carries the same energy (Listing 1:
// one Ehit per layer loop), so the per-task integer count n and one FP32
// product per task give a result that does not depend on the order in which
// hits were processed: the run-to-run reproducible counterpart of the
// paper's atomicAdd accumulation (Sec. 4, Listing 2).
//
// Record layout (uint64): [ cell | task | count - 1 (5 bits) ], with cell the
// index into the accumulation rows (row * acc_stride + cell in row).  The hit
// kernel writes the records to slots handed out in chunks (unused slots hold
// the empty record, all ones) and counts the records of every cell in the
// accumulation rows, used as uint32 counters.  Then:
//   1. an exclusive scan of the counters gives each cell the start of its
//      segment of the record array (int32) and zeroes the counters (calls of
//      sparse events: k_det_alloc, over the marked groups of 64 cells only);
//   2. scatter: every record takes a place in its cell's segment from the
//      cell's offset, counted up, which ends at the segment's end (the next
//      cell's start), so that one array bounds every segment.  In the
//      segment the cell is implied and a record shrinks to 32 bits:
//      [ task - first task of the cell's event (27 bits) | count - 1 ]
//      (a row holds one event, and its tasks are consecutive), so the
//      segments take half the bytes and sort as 32-bit keys;
//   3. fold: one thread per cell sorts its segment by (task, count) - a copy
//      in registers with a sorting network of 8, 16 or 32 records, each class
//      in a kernel of its own - merges the records of a task (their counts
//      add exactly) and folds; a warp per longer segment sorts it in shared
//      memory (bitonic) before its first lane folds.  The float result goes
//      to the (FP64) accumulation row, where the compaction of the atomic
//      mode picks it up, rounds it back to the same float and re-zeroes it.
// Only the order of places inside a segment depends on scheduling, and the
// sort removes it, so the cells are bit-reproducible.
#include <algorithm>
#include <atomic>

#include "fcs_internal.cuh"

namespace fcs {
namespace {

constexpr uint64_t kEmpty = ~0ull;
constexpr int kThreadSortMax = 32;  // segments sorted by one thread (in registers) up to here
constexpr int kRelTaskBits = 32 - kRecordCountBits;  // a segment record's task, relative to its event's first
constexpr uint32_t kCountMask = (1u << kRecordCountBits) - 1u;

// The first task of each event (row) of the range, from the per-particle task
// offsets: base[r] = poff[first particle of event ev_lo + r].
__global__ void k_det_bases(const int64_t* __restrict__ event_offsets, int32_t ev_lo, int32_t rows,
                            const int64_t* __restrict__ poff, const Sizes* sz, int64_t* __restrict__ base) {
  dependent_start();
  const int64_t n_part = sz->n_part, n_tasks = sz->n_tasks;
  const int64_t p0 = event_offsets[ev_lo];
  for (int32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
    const int64_t li = event_offsets[ev_lo + r] - p0;
    base[r] = (li >= 0 && li < n_part) ? poff[li] : n_tasks;  // events without particles take no records
  }
}

// A range that outgrew the workspace (FCS_FLAG_HIT_CAPACITY) has slots the
// hit kernel did not write: the scatter and the fold then do nothing (the
// call reports the overflow; the counter scan has zeroed the rows).
// A record whose task lies 2^27 or more past its event's first sets
// FCS_FLAG_KEY_BITS and is dropped (the call then fails).
__global__ void __launch_bounds__(256) k_det_scatter(const uint64_t* __restrict__ slots, Sizes* sz, int64_t cap,
                                                     int cell_shift, uint64_t task_mask, int32_t* __restrict__ cell_off,
                                                     int64_t n_cells_all, uint32_t acc_stride,
                                                     const int64_t* __restrict__ base, uint32_t* __restrict__ out) {
  dependent_start();
  if (sz->flags & FCS_FLAG_HIT_CAPACITY) return;
  constexpr int R = 4;  // records per thread and trip: their counts-up are in flight together
  const int64_t n = min(sz->n_slots, cap);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += R * stride) {
    uint64_t k[R];
#pragma unroll
    for (int j = 0; j < R; ++j) k[j] = (i0 + j * stride < n) ? slots[i0 + j * stride] : kEmpty;
    int32_t pos[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const uint64_t c = k[j] >> cell_shift;
      // (c is always in range for records of this range)
      pos[j] = (k[j] != kEmpty && c < (uint64_t)n_cells_all) ? atomicAdd(cell_off + c, 1) : -1;
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      if (pos[j] < 0) continue;
      const uint32_t c = (uint32_t)(k[j] >> cell_shift);
      const int64_t rel = (int64_t)((k[j] >> kRecordCountBits) & task_mask) - base[c / acc_stride];
      if (rel < 0 || rel >= ((int64_t)1 << kRelTaskBits)) {
        atomicOr(&sz->flags, (uint32_t)FCS_FLAG_KEY_BITS);
        continue;
      }
      if (pos[j] < cap) out[pos[j]] = ((uint32_t)rel << kRecordCountBits) | ((uint32_t)k[j] & kCountMask);
    }
  }
}

// Segment starts of the marked cells (calls of sparse events), in place of the
// scan over every counter: where a segment lies does not matter to the fold, so
// a warp adds up the records of the marked 64-cell groups among 128 and takes a
// run for them by one atomic, lists the groups for the fold, and leaves each
// group's start (gbase) beside its cells' ends.  Reads the marks and the marked
// counters; 500 single electrons' whole deterministic call 942 to 153 us.
constexpr int kAllocWarps = 8;
constexpr int kAllocGroups = 128;  // 4 marks to a lane
__global__ void __launch_bounds__(32 * kAllocWarps) k_det_alloc(const uint8_t* __restrict__ marks, int64_t n_groups,
                                                                uint32_t* __restrict__ counters,
                                                                int32_t* __restrict__ cell_off,
                                                                int32_t* __restrict__ gbase,
                                                                uint32_t* __restrict__ glist, Sizes* sz) {
  dependent_start();
  __shared__ uint16_t s_g[kAllocWarps][kAllocGroups];
  uint16_t* const list = s_g[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * kAllocWarps * kAllocGroups;
  for (int64_t g0 = ((int64_t)blockIdx.x * kAllocWarps + (threadIdx.x >> 5)) * kAllocGroups; g0 < n_groups; g0 += step) {
    const int64_t at = g0 + 4 * lane;
    uint32_t bits = 0;
    if (at + 4 <= n_groups) {
      const uint32_t m = *reinterpret_cast<const uint32_t*>(marks + at);
      bits = (m & 1u) | ((m >> 7) & 2u) | ((m >> 14) & 4u) | ((m >> 21) & 8u);
    } else {
      for (int j = 0; at + j < n_groups; ++j) bits |= (uint32_t)(marks[at + j] & 1u) << j;
    }
    int incl = __popc(bits);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int n = __shfl_sync(0xffffffffu, incl, 31);
    if (n == 0) continue;
    for (int p = incl - __popc(bits); bits; bits &= bits - 1u) list[p++] = (uint16_t)(4 * lane + __ffs(bits) - 1);
    __syncwarp();
    uint2* const cnt = reinterpret_cast<uint2*>(counters) + g0 * 32 + lane;
    int2* const off = reinterpret_cast<int2*>(cell_off) + g0 * 32 + lane;
    uint32_t sum = 0;
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      const uint2 v = cnt[32 * list[k]];
      sum += v.x + v.y;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    unsigned long long first = 0;
    if (lane == 0) first = atomicAdd(&sz->seg_alloc, ((unsigned long long)n << 32) | sum);
    first = __shfl_sync(0xffffffffu, first, 0);
    uint32_t run = (uint32_t)first;
    uint32_t* const gl = glist + (first >> 32);
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
      const int q = list[k];
      const uint2 v = cnt[32 * q];
      uint32_t x = v.x + v.y;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      const uint32_t a = run + x - v.x - v.y;
      off[32 * q] = make_int2((int32_t)a, (int32_t)(a + v.x));
      cnt[32 * q] = make_uint2(0u, 0u);
      if (lane == 0) {
        gbase[g0 + q] = (int32_t)run;
        gl[k] = (uint32_t)(g0 + q);
      }
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    __syncwarp();  // the list is reused
  }
}

__device__ __forceinline__ void sift_down(uint32_t* a, int64_t root, int64_t n) {
  while (true) {
    int64_t child = 2 * root + 1;
    if (child >= n) return;
    if (child + 1 < n && a[child + 1] > a[child]) ++child;
    if (a[root] >= a[child]) return;
    const uint32_t t = a[root];
    a[root] = a[child];
    a[child] = t;
    root = child;
  }
}

// Ascending sort of a[0, n) in place (heapsort).
__device__ __noinline__ void sort_segment(uint32_t* a, int64_t n) {
  for (int64_t r = n / 2 - 1; r >= 0; --r) sift_down(a, r, n);
  for (int64_t e = n - 1; e > 0; --e) {
    const uint32_t t = a[0];
    a[0] = a[e];
    a[e] = t;
    sift_down(a, 0, e);
  }
}

// One step of the fold of a cell's records in ascending order: per task the
// summed count times the task's hit energy, added in task order.  The count
// is 32-bit (a task's hits fit in 31 bits) and converted as such: conversions
// from 64-bit integers, like float-to-double ones, run on the narrow FP64 pipe.
struct Fold {
  float E = 0.0f;
  float e = 0.0f;  // hit energy of prev_task
  int64_t prev_task = -1;  // relative to the event's first task
  uint32_t cnt = 0;
  // segment record k, whose task's hit energy is ek (loaded ahead by the caller)
  __device__ __forceinline__ void add(uint32_t k, float ek) {
    const int64_t task = (int64_t)(k >> kRecordCountBits);
    const uint32_t c = (k & kCountMask) + 1u;
    if (task != prev_task) {
      if (prev_task >= 0) E = __fadd_rn(E, __fmul_rn((float)cnt, e));
      prev_task = task;
      e = ek;
      cnt = 0;
    }
    cnt += c;
  }
  // segment record k, the task's hit energy read from the event's part of
  // the table when the task changes
  __device__ __forceinline__ void add(uint32_t k, const float* __restrict__ ev_ehit) {
    const int64_t task = (int64_t)(k >> kRecordCountBits);
    const uint32_t c = (k & kCountMask) + 1u;
    if (task != prev_task) {
      if (prev_task >= 0) E = __fadd_rn(E, __fmul_rn((float)cnt, e));
      prev_task = task;
      e = ev_ehit[task];
      cnt = 0;
    }
    cnt += c;
  }
  // the folded float, as the FP64 row value the compaction reads (an exact
  // widening done with integer operations)
  __device__ __forceinline__ double result() const { return f32_to_f64_bits(__fadd_rn(E, __fmul_rn((float)cnt, e))); }
};

// Ascending sort of N keys in registers (N a power of two): Batcher's
// odd-even merge sort (Batcher 1968; 19 compare-exchanges for 8 keys, 63 for
// 16), every index a compile-time constant; absent records are all ones and
// sort last.
__device__ __forceinline__ void cmpx(uint32_t& x, uint32_t& y) {
  const uint32_t lo = min(x, y), hi = max(x, y);
  x = lo;
  y = hi;
}

// Merge of the sorted halves of r[LO, LO + N) taken with stride R: the odd
// and even subsequences recursively, then neighbours R apart.
template <int LO, int N, int R, int M>
__device__ __forceinline__ void oe_merge(uint32_t (&r)[M]) {
  constexpr int S = 2 * R;
  if constexpr (S < N) {
    oe_merge<LO, N, S>(r);
    oe_merge<LO + R, N, S>(r);
#pragma unroll
    for (int i = LO + R; i + R < LO + N; i += S) cmpx(r[i], r[i + R]);
  } else {
    cmpx(r[LO], r[LO + R]);
  }
}
template <int LO, int N, int M>
__device__ __forceinline__ void oe_sort(uint32_t (&r)[M]) {
  if constexpr (N > 1) {
    oe_sort<LO, N / 2>(r);
    oe_sort<LO + N / 2, N / 2>(r);
    oe_merge<LO, N, 1>(r);
  }
}
template <int N>
__device__ __forceinline__ void merge_sort_net(uint32_t (&r)[N]) {
  oe_sort<0, N>(r);
}

// Sort and fold of a segment of n <= N records (a register copy).  The hit
// energies of the sorted records' tasks are loaded all at once, ahead of the
// fold, so that the cell waits for one load latency, not one per task.
template <int N>
__device__ __forceinline__ double fold_small(const uint32_t* __restrict__ recs, int64_t a, int n,
                                            const float* __restrict__ ev_ehit) {
  uint32_t r[N];
#pragma unroll
  for (int j = 0; j < N; ++j) r[j] = j < n ? recs[a + j] : ~0u;
  merge_sort_net<N>(r);
  float e[N];
#pragma unroll
  for (int j = 0; j < N; ++j) e[j] = j < n ? ev_ehit[r[j] >> kRecordCountBits] : 0.0f;
  Fold f;
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (j < n) f.add(r[j], e[j]);
  return f.result();
}

// Cell c's segment [a, b) after the scatter: cell_off[c] holds its end, which
// is the next cell's start (of its group, with gbase).
__device__ __forceinline__ void segment(const int32_t* __restrict__ cell_off, const int32_t* __restrict__ gbase,
                                        int64_t c, int64_t cap, int64_t& a, int64_t& b) {
  a = gbase && (c & 63) == 0 ? gbase[c >> 6] : (c > 0 ? cell_off[c - 1] : 0);
  b = min((int64_t)cell_off[c], cap);
}

// The hit energies of the tasks of cell c's event.
__device__ __forceinline__ const float* event_ehit(const float* __restrict__ task_ehit,
                                                  const int64_t* __restrict__ base, int64_t c, uint32_t acc_stride) {
  return task_ehit + base[(uint32_t)c / acc_stride];
}

// Segments of up to 8 records (92 % of the hit cells of pile-up events) are
// sorted as a copy in registers, with nothing written back, and folded;
// segments of 9 to 16 and of 17 to kThreadSortMax records are listed for the
// two k_det_fold_mid kernels and longer ones for k_det_fold_big, so that the
// warps of each kernel run one path.  The list array holds three lists, from
// its start, a third in and two thirds in: a listed cell has at least 9 records,
// so each list fits its third.
//
// Most cells are empty (half of a pile-up event's, 95 % of a hard scatter's),
// and a warp that folds 32 neighbouring cells folds for the few that are not.
// So a warp reads the offsets of 64 cells at a time, puts the cells to fold into
// a queue of its own and folds 32 of them whenever it holds that many: 33 hard
// scatters 52 to 26 us, the whole call of 64 pile-up events 1478 to 1431 (256
// cells at a time, 5 CTAs per SM: 28 us and 1446).
constexpr int kFoldWarps = 8, kFoldLoads = 2;
constexpr int kFoldQueue = 32 * (kFoldLoads + 1);  // < 32 left after the folds + the new

struct FoldEnt {
  uint32_t c;     // cell
  int32_t a, n;   // its segment
};

// SPARSE: the cells of the listed groups of 64 only.
template <bool SPARSE>
__global__ void __launch_bounds__(32 * kFoldWarps, 6) k_det_fold(const uint32_t* __restrict__ recs,
                                                  const int32_t* __restrict__ cell_off, int64_t n_cells_all, Sizes* sz,
                                                  int64_t cap, uint32_t acc_stride, const int64_t* __restrict__ base,
                                                  const float* __restrict__ task_ehit, double* __restrict__ acc,
                                                  int64_t* __restrict__ lists, const int32_t* __restrict__ gbase,
                                                  const uint32_t* __restrict__ glist) {
  dependent_start();
  __shared__ FoldEnt s_q[kFoldWarps][kFoldQueue];
  if (sz->flags & (FCS_FLAG_HIT_CAPACITY | FCS_FLAG_KEY_BITS)) return;
  const int lane = threadIdx.x & 31;
  FoldEnt* const queue = s_q[threadIdx.x >> 5];
  const unsigned below = (1u << lane) - 1u;
  int held = 0;
  static_assert(32 * kFoldLoads == 64, "a trip is a group of marked cells");
  const int64_t n_trips = SPARSE ? (int64_t)(sz->seg_alloc >> 32) : (n_cells_all + 63) / 64;
  const int64_t step = (int64_t)gridDim.x * kFoldWarps;
  // warp-uniform trips, so that the lists take one counter update per warp
  for (int64_t q = (int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5); q < n_trips; q += step) {
    const int64_t w0 = 64 * (SPARSE ? (int64_t)glist[q] : q);
    // the segment ends (int32, as is the record count) and the one before the
    // warp's first cell
    int32_t ends[kFoldLoads];
#pragma unroll
    for (int j = 0; j < kFoldLoads; ++j) {
      const int64_t c = w0 + 32 * j + lane;
      ends[j] = c < n_cells_all ? cell_off[c] : -1;
    }
    int32_t prev = SPARSE ? gbase[w0 >> 6] : (w0 > 0 ? cell_off[w0 - 1] : 0);  // the end before the row of 32
#pragma unroll
    for (int j = 0; j < kFoldLoads; ++j) {
      const int64_t c = w0 + 32 * j + lane;
      const int32_t up = __shfl_up_sync(0xffffffffu, ends[j], 1);
      const int32_t a = lane ? up : prev;
      prev = __shfl_sync(0xffffffffu, ends[j], 31);
      const int32_t n = ends[j] >= 0 ? (int32_t)(min((int64_t)ends[j], cap) - a) : 0;
      if (!__any_sync(0xffffffffu, n > 0)) continue;
      const unsigned mb = __ballot_sync(0xffffffffu, n > kThreadSortMax);
      const unsigned m16 = __ballot_sync(0xffffffffu, n > 8 && n <= 16);
      const unsigned m32 = __ballot_sync(0xffffffffu, n > 16 && n <= kThreadSortMax);
      if (mb | m16 | m32) {
        unsigned long long bb = 0, b16 = 0, b32 = 0;
        if (lane == 0) {
          if (mb) bb = atomicAdd((unsigned long long*)&sz->n_big, (unsigned long long)__popc(mb));
          if (m16) b16 = atomicAdd((unsigned long long*)&sz->n_mid, (unsigned long long)__popc(m16));
          if (m32) b32 = atomicAdd((unsigned long long*)&sz->n_mid32, (unsigned long long)__popc(m32));
        }
        bb = __shfl_sync(0xffffffffu, bb, 0);
        b16 = __shfl_sync(0xffffffffu, b16, 0);
        b32 = __shfl_sync(0xffffffffu, b32, 0);
        if ((mb >> lane) & 1u) lists[bb + __popc(mb & below)] = c;
        if ((m16 >> lane) & 1u) lists[cap / 3 + (int64_t)(b16 + __popc(m16 & below))] = c;
        if ((m32 >> lane) & 1u) lists[2 * (cap / 3) + (int64_t)(b32 + __popc(m32 & below))] = c;
      }
      const bool small = n > 0 && n <= 8;
      const unsigned ms = __ballot_sync(0xffffffffu, small);
      if (small) queue[held + __popc(ms & below)] = FoldEnt{(uint32_t)c, a, n};
      held += __popc(ms);
    }
#pragma unroll 1
    while (held >= 32 || (held && q + step >= n_trips)) {  // (the last trip folds what is left)
      const int cnt = min(held, 32);
      __syncwarp();
      if (lane < cnt) {
        const FoldEnt e = queue[held - cnt + lane];
        acc[e.c] = fold_small<8>(recs, e.a, e.n, event_ehit(task_ehit, base, e.c, acc_stride));
      }
      held -= cnt;
    }
    __syncwarp();
  }
}

// One thread per listed cell of 9 to 16 (N = 16) or 17 to 32 records
// (N = 32): sorted as a copy in registers, then folded.
template <int N>
__global__ void __launch_bounds__(256) k_det_fold_mid(const uint32_t* __restrict__ recs,
                                                      const int32_t* __restrict__ cell_off, int64_t n_cells_all,
                                                      const Sizes* sz, int64_t cap, uint32_t acc_stride,
                                                      const int64_t* __restrict__ base,
                                                      const float* __restrict__ task_ehit, double* __restrict__ acc,
                                                      const int64_t* __restrict__ lists,
                                                      const int32_t* __restrict__ gbase) {
  dependent_start();
  static_assert(N == 16 || N == kThreadSortMax, "two mid classes");
  if (sz->flags & (FCS_FLAG_HIT_CAPACITY | FCS_FLAG_KEY_BITS)) return;
  const int64_t n_list = N == 16 ? sz->n_mid : sz->n_mid32;
  const int64_t* list = lists + (N == 16 ? cap / 3 : 2 * (cap / 3));
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n_list; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = list[q];
    int64_t a, b;
    segment(cell_off, gbase, c, cap, a, b);
    acc[c] = fold_small<N>(recs, a, (int)(b - a), event_ehit(task_ehit, base, c, acc_stride));
  }
}

// One warp per long segment.  Its records are many and their tasks few (a task
// leaves a record per warp step), so the warp first sums the counts by task in a
// hash table in shared memory, then sorts the tasks (bitonic) and lane 0 adds
// their products.  (Sorting the records, 33 hard scatters' whole call took 291
// us, 281 so; 64 events of four 1 TeV electrons, whose cores hold more than 1024
// records a cell, by heapsort 2330 us, 450 so; of 4 TeV 16.2 and 1.3 ms.)
// Segments of more tasks than the table takes are sorted record by record: in
// shared memory up to kBigMax of them, longer ones by heapsort in place.
constexpr int kBigWarps = 4;
constexpr int kBigMax = 1024;
constexpr int kBigSlots = 512;                // of the table
constexpr int kBigTasks = kBigSlots * 3 / 4;  // it takes

// Slot of a task in the table (linear probing; at least a quarter is empty
// while no more than kBigTasks tasks and 32 lanes' insertions are in, so the
// search ends).
__device__ __forceinline__ int task_slot(uint32_t task) { return (int)((task * 2654435761u) >> 23); }

// Sorts the m keys (a power of two) of one warp, ascending.
__device__ __forceinline__ void warp_bitonic(uint32_t* s, int m, int lane) {
  for (int k = 2; k <= m; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int i = lane; i < m; i += 32) {
        const int l = i ^ jj;
        if (l > i) {
          const uint32_t x = s[i], y = s[l];
          const bool up = (i & k) == 0;
          if ((x > y) == up) {
            s[i] = y;
            s[l] = x;
          }
        }
      }
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(32 * kBigWarps) k_det_fold_big(uint32_t* __restrict__ recs,
                                                                 const int32_t* __restrict__ cell_off,
                                                                 int64_t n_cells_all, const Sizes* sz, int64_t cap,
                                                                 uint32_t acc_stride, const int64_t* __restrict__ base,
                                                                 const float* __restrict__ task_ehit,
                                                                 double* __restrict__ acc,
                                                                 const int64_t* __restrict__ big,
                                                                 const int32_t* __restrict__ gbase) {
  dependent_start();
  __shared__ uint32_t s_rec[kBigWarps][kBigMax];
  __shared__ float s_e[kBigWarps][kBigMax];  // the sorted records' hit energies
  if (sz->flags & (FCS_FLAG_HIT_CAPACITY | FCS_FLAG_KEY_BITS)) return;
  const int64_t n_big = sz->n_big;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  uint32_t* s = s_rec[wi];
  float* se = s_e[wi];
  for (int64_t q = (int64_t)blockIdx.x * kBigWarps + wi; q < n_big; q += (int64_t)gridDim.x * kBigWarps) {
    const int64_t c = big[q];
    int64_t a, b;
    segment(cell_off, gbase, c, cap, a, b);
    const int64_t n = b - a;
    uint32_t* seg = recs + a;
    const float* ev_ehit = event_ehit(task_ehit, base, c, acc_stride);
    // the table: tasks and counts; then the sorted tasks and their products
    volatile uint32_t* const key = s;
    uint32_t* const cnt = s + kBigSlots;
    uint32_t* const sorted = reinterpret_cast<uint32_t*>(se);
    float* const prod = se + kBigSlots;
    for (int j = lane; j < kBigSlots; j += 32) {
      key[j] = ~0u;
      cnt[j] = 0;
    }
    __syncwarp();
    int tasks = 0;
    for (int64_t j0 = 0; j0 < n && tasks <= kBigTasks - 32; j0 += 32) {
      bool fresh = false;
      if (j0 + lane < n) {
        const uint32_t k = seg[j0 + lane], task = k >> kRecordCountBits;
        int h = task_slot(task);
        while (key[h] != task) {
          const uint32_t was = key[h] == ~0u ? atomicCAS(s + h, ~0u, task) : key[h];
          if (was == ~0u) fresh = true;
          if (was == ~0u || was == task) break;
          h = (h + 1) & (kBigSlots - 1);
        }
        atomicAdd(cnt + h, (k & kCountMask) + 1u);
      }
      tasks += __popc(__ballot_sync(0xffffffffu, fresh));
    }
    if (tasks <= kBigTasks - 32) {
      __syncwarp();
      int at = 0;
      for (int j0 = 0; j0 < kBigSlots; j0 += 32) {
        const uint32_t k = key[j0 + lane];
        const unsigned m = __ballot_sync(0xffffffffu, k != ~0u);
        if (k != ~0u) sorted[at + __popc(m & ((1u << lane) - 1u))] = k;
        at += __popc(m);
      }
      int m = 1;
      while (m < tasks) m <<= 1;
      for (int j = tasks + lane; j < m; j += 32) sorted[j] = ~0u;
      __syncwarp();
      warp_bitonic(sorted, m, lane);
      for (int j = lane; j < tasks; j += 32) {
        const uint32_t task = sorted[j];
        int h = task_slot(task);
        while (key[h] != task) h = (h + 1) & (kBigSlots - 1);
        prod[j] = __fmul_rn((float)cnt[h], ev_ehit[task]);
      }
      __syncwarp();
      if (lane == 0) {
        float E = 0.0f;
        for (int j = 0; j < tasks; ++j) E = __fadd_rn(E, prod[j]);
        acc[c] = f32_to_f64_bits(E);
      }
      __syncwarp();
      continue;
    }
    __syncwarp();
    if (n > kBigMax) {
      if (lane == 0) {
        sort_segment(seg, n);
        Fold f;
        for (int64_t j = 0; j < n; ++j) f.add(seg[j], ev_ehit);
        acc[c] = f.result();
      }
      __syncwarp();
      continue;
    }
    int m = 1;
    while (m < n) m <<= 1;
    for (int j = lane; j < m; j += 32) s[j] = j < n ? seg[j] : ~0u;
    __syncwarp();
    warp_bitonic(s, m, lane);
    // the hit energies, loaded by all lanes at once; then the first lane folds
    for (int j = lane; j < n; j += 32) se[j] = ev_ehit[s[j] >> kRecordCountBits];
    __syncwarp();
    if (lane == 0) {
      Fold f;
      for (int64_t j = 0; j < n; ++j) f.add(s[j], se[j]);
      acc[c] = f.result();
    }
    __syncwarp();
  }
}

constexpr int kMaxDevices = 64;

// Blocks of 256 threads of k_det_fold that one SM holds at once (per device,
// looked up once): the kernel loops grid-stride, and a grid beyond one wave of
// resident blocks would run its surplus as a second, mostly empty wave.
int fold_resident_blocks() {
  static std::atomic<int> occ_by_device[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = kMaxDevices - 1;
  int occ = occ_by_device[dev].load(std::memory_order_relaxed);
  if (!occ) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_det_fold<false>, 256, 0) != cudaSuccess) {
      (void)cudaGetLastError();
      occ = 1;
    }
    occ = std::max(occ, 1);
    occ_by_device[dev].store(occ, std::memory_order_relaxed);
  }
  return occ;
}

}  // namespace

cudaError_t launch_det_reduce(const GeoDev& g, WsDev w, int32_t rows, int key_task_bits, int64_t* scratch,
                              const int64_t* event_offsets, int32_t ev_lo, ScanTmp tmp, const Launch& L) {
  const int64_t n_cells_all = (int64_t)rows * g.acc_stride;
  uint32_t* counters = reinterpret_cast<uint32_t*>(w.acc);
  int64_t* base = scratch;                                       // [rows] first task of each event
  int32_t* cell_off = reinterpret_cast<int32_t*>(scratch + rows);  // [n_cells_all] segment starts, then ends
  const uint32_t stride = (uint32_t)g.acc_stride;
  cudaError_t e = launch_dependent(k_det_bases, (rows + 255) / 256, 256, 0, L.s, event_offsets, ev_lo, rows, w.poff,
                                   w.sizes, base);
  if (e != cudaSuccess) return e;
  // the scratch holds 8 bytes per cell: the offsets' are followed by the groups'
  const int64_t n_groups = n_cells_all >> kMarkShift;
  int32_t* gbase = w.marks ? cell_off + n_cells_all : nullptr;          // [n_groups]
  uint32_t* glist = reinterpret_cast<uint32_t*>(cell_off + n_cells_all) + n_groups;  // [marked groups]
  if (w.marks) {
    const int64_t ctas = (n_groups + kAllocWarps * kAllocGroups - 1) / (kAllocWarps * kAllocGroups);
    e = launch_dependent(k_det_alloc, std::min<int64_t>(ctas, L.num_sms * 8), 32 * kAllocWarps, 0, L.s, w.marks, n_groups,
                         counters, cell_off, gbase, glist, w.sizes);
  } else {
    e = launch_scan_u32_zero(counters, cell_off, n_cells_all, tmp, L.s);
  }
  if (e != cudaSuccess) return e;
  const int cell_shift = kRecordCountBits + key_task_bits;
  const uint64_t task_mask = (key_task_bits >= 64) ? ~0ull : ((1ull << key_task_bits) - 1ull);
  uint32_t* segs = reinterpret_cast<uint32_t*>(w.keys_alt);
  e = launch_dependent(k_det_scatter, L.num_sms * 8, 256, 0, L.s, w.keys, w.sizes, w.rec_cap, cell_shift, task_mask,
                       cell_off, n_cells_all, stride, base, segs);
  if (e != cudaSuccess) return e;
  // the slot array is free after the scatter: it lists the segments of more
  // than 8 records
  int64_t* lists = reinterpret_cast<int64_t*>(w.keys);
  const int64_t fold_grid = (int64_t)L.num_sms * fold_resident_blocks();
  e = launch_dependent(w.marks ? k_det_fold<true> : k_det_fold<false>, fold_grid, 256, 0, L.s, segs, cell_off, n_cells_all,
                       w.sizes, w.rec_cap, stride, base, w.tehit, w.acc, lists, gbase, glist);
  if (e != cudaSuccess) return e;
  e = launch_dependent(k_det_fold_mid<16>, L.num_sms * 4, 256, 0, L.s, segs, cell_off, n_cells_all, w.sizes, w.rec_cap,
                       stride, base, w.tehit, w.acc, lists, gbase);
  if (e != cudaSuccess) return e;
  e = launch_dependent(k_det_fold_mid<kThreadSortMax>, L.num_sms * 2, 256, 0, L.s, segs, cell_off, n_cells_all, w.sizes,
                       w.rec_cap, stride, base, w.tehit, w.acc, lists, gbase);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_det_fold_big, L.num_sms * 4, 32 * kBigWarps, 0, L.s, segs, cell_off, n_cells_all, w.sizes,
                          w.rec_cap, stride, base, w.tehit, w.acc, lists, gbase);
}

}  // namespace fcs
