// fcs_compact.cu - gathers the hit cells of each event as (cell id, E) pairs
// for the transfer of results (the paper's sim_ct kernel, Sec. 4) and resets
// the accumulation rows to zero in the same pass (the paper's separate
// clean kernel, Sec. 4, is folded in).  The rows are FP64 (fcs_internal.cuh:
// acc_add); each hit cell is rounded once to the float of the output.
// Output order: event-major, ascending
// cell id; each chunk's output offset is the count of the chunks before it,
// taken in one pass by a decoupled look-back, so the result is deterministic
// and the rows are read once.
#include "fcs_internal.cuh"
#include "fcs_lookback.cuh"

namespace fcs {
namespace {

constexpr int kCThreads = 256;
constexpr int kCWarps = kCThreads / 32;
constexpr int kCRows = 8;               // 64-cell rows of a warp's share (rows are padded to 64 cells)
constexpr int kShare = 64 * kCRows;
constexpr int kChunk = kCWarps * kShare;  // 4096 cells
constexpr int kCtasPerSm = 4;

// A row value is a hit cell when it is not +-0 (an integer test, off the FP64 pipe).
__device__ __forceinline__ bool acc_nonzero(double d) {
  return ((unsigned long long)__double_as_longlong(d) << 1) != 0ull;
}

struct CompactArgs {
  double* acc;
  int32_t n_cells, stride, cpr, ev_lo;
  int32_t one_run;
  int64_t n_chunks;
  uint64_t* state;
  int64_t cap_tiles;
  uint32_t* flags;
  int64_t* total_dst;
  float* cells_out;
  int32_t* cell_ids;
  float* cell_E;
  int64_t* event_offsets_out;
  int64_t capacity;
};

// One pass over the chunks: CTAs take them in ticket order; a chunk packs its
// hit cells into shared memory as it reads them, publishes their count, looks
// back for the count of the chunks before it (the first chunk starts at
// *total_dst, the call's running output size) and writes its pairs; the last
// chunk leaves the new total in *total_dst.  The last CTA to finish resets the
// ticket and the status words.  A chunk's ticket is taken when the chunk before
// it is written: a chunk held while its CTA still looks back publishes nothing,
// and every look-back behind it waits (1024 events: 3270 us).
//
// Bound by memory (the rows in, the pairs out, the zeros) and by the look-backs:
// 32 chunks in half a microsecond.  A warp takes 512 consecutive cells, 64 to
// an instruction, 16 bytes a lane, all eight rows in flight at once; places in
// the output come from ballots.  Compaction of 500 single electrons (753 MB of
// nearly empty rows), 64 and 1024 pile-up events (1.5 GB of rows, 95M pairs):
//   387, 78 and 960 us   each lane 16 consecutive cells, places by a block scan
//   275, 65 and 795      here
//   248, 74 and 866      8192-cell chunks (before the warps wrote by themselves)
//   369, 100 and 1356    chunks by bulk copy into shared memory, three in
//                        flight a CTA (its tickets are held)
// DENSE: also the dense rows.  PAIRS: the pairs are wanted (else their number).
template <bool DENSE, bool PAIRS>
__global__ void __launch_bounds__(kCThreads, kCtasPerSm) k_compact_one(const CompactArgs A) {
  dependent_start();
  __shared__ float s_E[PAIRS ? kChunk : 1];
  __shared__ uint16_t s_at[PAIRS ? kChunk : 1];  // place in the chunk
  __shared__ int s_w[kCWarps];
  __shared__ unsigned long long s_ticket;
  __shared__ int64_t s_base;
  __shared__ int s_last;
  unsigned long long* ticket = reinterpret_cast<unsigned long long*>(A.state);
  unsigned long long* done = ticket + 1;
  uint64_t* status = A.state + 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned below = (1u << lane) - 1u;
  int64_t n_t = A.n_chunks;
  if (n_t > A.cap_tiles) {  // the workspace sizes the state for its chunks: never
    if (tid == 0) atomicOr(A.flags, (uint32_t)FCS_FLAG_WAIT_TIMEOUT);
    n_t = 0;
  }
  while (true) {
    if (tid == 0) s_ticket = atomicAdd(ticket, 1ull);
    __syncthreads();
    const int64_t t = (int64_t)s_ticket;
    if (t >= n_t) break;
    const int64_t row = t / A.cpr;
    const int cc = (int)(t % A.cpr) * kChunk;  // the chunk's first cell in its row
    const int c0 = cc + warp * kShare;         // the warp's
    const int rows = min(kCRows, max(0, (A.stride - c0) / 64));
    double2* const src = reinterpret_cast<double2*>(A.acc + row * A.stride + c0) + lane;
    float* const dense = DENSE ? A.cells_out + (int64_t)(A.ev_lo + row) * A.n_cells : nullptr;
    int n = 0;  // the warp's hit cells
    double2 v[kCRows];
#pragma unroll
    for (int j = 0; j < kCRows; ++j) v[j] = j < rows ? src[32 * j] : make_double2(0.0, 0.0);
#pragma unroll
    for (int j = 0; j < kCRows; ++j) {
      const bool nx = acc_nonzero(v[j].x), ny = acc_nonzero(v[j].y);
      const unsigned mx = __ballot_sync(0xffffffffu, nx), my = __ballot_sync(0xffffffffu, ny);
      float fx = 0.0f, fy = 0.0f;
      if (mx | my) {
        if (nx || ny) src[32 * j] = make_double2(0.0, 0.0);  // re-zero what is not zero
        if (DENSE || PAIRS) {
          fx = acc_to_f32(v[j].x);
          fy = acc_to_f32(v[j].y);
        }
        if constexpr (PAIRS) {
          const int p = warp * kShare + n + __popc(mx & below) + __popc(my & below);
          const int at = warp * kShare + 64 * j + 2 * lane;
          if (nx) {
            s_E[p] = fx;
            s_at[p] = (uint16_t)at;
          }
          if (ny) {
            s_E[p + (nx ? 1 : 0)] = fy;
            s_at[p + (nx ? 1 : 0)] = (uint16_t)(at + 1);
          }
        }
        n += __popc(mx) + __popc(my);
      }
      if constexpr (DENSE) {
        const int c = c0 + 64 * j + 2 * lane;
        if (j < rows) {
          if ((A.n_cells & 1) == 0) {  // then c is even and in the row with c + 1
            if (c < A.n_cells) *reinterpret_cast<float2*>(dense + c) = make_float2(fx, fy);
          } else {
            if (c < A.n_cells) dense[c] = fx;
            if (c + 1 < A.n_cells) dense[c + 1] = fy;
          }
        }
      }
    }
    if (lane == 0) s_w[warp] = n;
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int w = 0; w < kCWarps; ++w) total += s_w[w];
    if (warp == 0) {  // publish, look back, publish the prefix
      int64_t excl;
      if (t == 0) {
        excl = *A.total_dst;
      } else {
        if (lane == 0) atomicExch(reinterpret_cast<unsigned long long*>(status + t), kFlagAgg | (uint64_t)total);
        excl = look_back(status, t, A.flags);
      }
      if (lane == 0) {
        atomicExch(reinterpret_cast<unsigned long long*>(status + t), kFlagPrefix | (uint64_t)(excl + total));
        s_base = excl;
        if (t % A.cpr == 0 && A.event_offsets_out) A.event_offsets_out[A.ev_lo + row] = excl;
        if (t == n_t - 1) *A.total_dst = excl + total;
      }
    }
    __syncthreads();
    if constexpr (PAIRS) {
      int pre[kCWarps];  // the warps' first pairs in the chunk
      pre[0] = 0;
#pragma unroll
      for (int w = 1; w < kCWarps; ++w) pre[w] = pre[w - 1] + s_w[w - 1];
      const int64_t pos = s_base;
      const int m = (int)max((int64_t)0, min((int64_t)total, A.capacity - pos));
      if (A.one_run) {
        // a chunk's pairs as one run (into host memory, over the link: 64
        // events end to end 1345 us, warp by warp 1370)
        for (int q = tid; q < m; q += kCThreads) {
          int first = 0, w = 0;
#pragma unroll
          for (int k = 1; k < kCWarps; ++k) {
            if (q >= pre[k]) {
              first = pre[k];
              w = k;
            }
          }
          const int at = w * kShare + q - first;
          A.cell_ids[pos + q] = cc + s_at[at];
          A.cell_E[pos + q] = s_E[at];
        }
      } else {
        // each warp its own (into device memory: 1024 events 795 us, as one run 846)
        int first = 0;
#pragma unroll
        for (int k = 1; k < kCWarps; ++k) first = warp == k ? pre[k] : first;
        for (int q = lane; q < n && first + q < m; q += 32) {
          A.cell_ids[pos + first + q] = cc + s_at[warp * kShare + q];
          A.cell_E[pos + first + q] = s_E[warp * kShare + q];
        }
      }
      __syncthreads();  // the shared arrays are reused
    }
  }
  // every CTA has left its loop (and its look-backs) before it counts itself
  // done; the last one resets the state
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1ull) == (unsigned long long)gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int64_t i = tid; i < n_t; i += kCThreads) status[i] = 0;
    if (tid == 0) {
      *ticket = 0;
      *done = 0;
    }
  }
}

constexpr int kSparseCtas = 8;       // per SM
constexpr int kSparseParts = 304;    // parts wanted of all rows

// Rows of sparse events (some particles each): a CTA takes a part of a row (all
// of it from 304 rows on), in ticket order, lists the 64-cell groups that the
// range's deposits marked there, gives each warp a run of them, and reads only
// those: once to count and again, from the caches and only where the run is
// too long for the warp's registers, to write the pairs and zero the cells.
//
// k_compact_one reads every row: 500 single electrons leave 27,782 hit cells in
// 753 MB, and the look-backs run over 23,000 chunks.  Here the marks (1.5 MB)
// and the marked groups are read, and the look-backs run over 500 parts; what
// is left is the chain ticket, marks, groups, look-back, pairs of one CTA.
// Rows x particles of 65 GeV:   16 x 1   64 x 1   500 x 1   500 x 8   16384 x 1
//   k_compact_one (us)            21       47       275       297       8600
//   here                          16       18        21        90        300
// (marks of 4096 cells 133 us at 500 x 1; parts for 608 CTAs of 4 an SM, 8
// groups in flight 25.)
// DENSE: also the dense rows, zeros first and the marked cells over them (500
// single electrons, the whole call: 387 us by k_compact_one, 179 here).
template <bool DENSE>
__global__ void __launch_bounds__(kCThreads, kSparseCtas) k_compact_sparse(const CompactArgs A, uint8_t* __restrict__ marks) {
  dependent_start();
  __shared__ uint16_t s_list[kMaxRowMarks];  // the part's marked groups, in order
  __shared__ int s_w[kCWarps];               // per warp: marked groups listed; then hit cells
  __shared__ unsigned long long s_ticket;
  __shared__ int64_t s_base;
  __shared__ int s_last;
  constexpr int kSeg = kMaxRowMarks / kCThreads;  // marks of a lane, at most
  constexpr int kLoads = 2;                       // groups of a warp in flight
  unsigned long long* ticket = reinterpret_cast<unsigned long long*>(A.state);
  unsigned long long* done = ticket + 1;
  uint64_t* status = A.state + 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned below = (1u << lane) - 1u;
  const int row_marks = A.stride >> kMarkShift;
  const int part_marks = (row_marks + A.cpr - 1) / A.cpr;
  const int seg = (part_marks + kCWarps - 1) / kCWarps;  // marks of a warp
  int64_t n_t = A.n_chunks;                              // parts
  if (n_t > A.cap_tiles) {  // the workspace sizes the state for more: never
    if (tid == 0) atomicOr(A.flags, (uint32_t)FCS_FLAG_WAIT_TIMEOUT);
    n_t = 0;
  }
  while (true) {
    if (tid == 0) s_ticket = atomicAdd(ticket, 1ull);
    __syncthreads();
    const int64_t t = (int64_t)s_ticket;
    if (t >= n_t) break;
    const int64_t row = t / A.cpr;
    const int mark0 = (int)(t % A.cpr) * part_marks;
    float* const dense = DENSE ? A.cells_out + (A.ev_lo + row) * (int64_t)A.n_cells : nullptr;
    if constexpr (DENSE) {  // (the barriers below order the zeros before the cells)
      const int c0 = mark0 << kMarkShift, c1 = min((mark0 + part_marks) << kMarkShift, A.n_cells);
      if ((A.n_cells & 3) == 0 && (reinterpret_cast<uintptr_t>(dense) & 15) == 0) {
        for (int c = c0 + 4 * tid; c < c1; c += 4 * kCThreads)
          *reinterpret_cast<float4*>(dense + c) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      } else {
        for (int c = c0 + tid; c < c1; c += kCThreads) dense[c] = 0.0f;
      }
    }
    double2* const cells = reinterpret_cast<double2*>(A.acc + row * A.stride) + lane;
    {
      const int first = mark0 + warp * seg;
      const int n = min(seg, min(mark0 + part_marks, row_marks) - first);
      uint8_t* const mine = marks + row * row_marks + first + lane;
      bool on[kSeg];
#pragma unroll
      for (int j = 0; j < kSeg; ++j) on[j] = 32 * j + lane < n && mine[32 * j] != 0;
      int cnt = 0;
#pragma unroll
      for (int j = 0; j < kSeg; ++j) {
        cnt += __popc(__ballot_sync(0xffffffffu, on[j]));
        if (on[j]) mine[32 * j] = 0;
      }
      if (lane == 0) s_w[warp] = cnt;
      __syncthreads();
      int at = 0;
      for (int w = 0; w < warp; ++w) at += s_w[w];
#pragma unroll
      for (int j = 0; j < kSeg; ++j) {
        const unsigned m = __ballot_sync(0xffffffffu, on[j]);
        if (on[j]) s_list[at + __popc(m & below)] = (uint16_t)(first + 32 * j + lane);
        at += __popc(m);
      }
    }
    int listed = 0;
#pragma unroll
    for (int w = 0; w < kCWarps; ++w) listed += s_w[w];
    __syncthreads();  // the list is written, s_w is read
    const int run = (listed + kCWarps - 1) / kCWarps;
    const int lo = warp * run, hi = min(listed, lo + run);
    double2 v[kLoads];
    auto load = [&](int k) {
#pragma unroll
      for (int j = 0; j < kLoads; ++j) v[j] = k + j < hi ? cells[32 * s_list[k + j]] : make_double2(0.0, 0.0);
    };
    int n = 0;  // the warp's hit cells
    for (int k = lo; k < hi; k += kLoads) {
      load(k);
#pragma unroll
      for (int j = 0; j < kLoads; ++j)
        n += __popc(__ballot_sync(0xffffffffu, acc_nonzero(v[j].x))) +
             __popc(__ballot_sync(0xffffffffu, acc_nonzero(v[j].y)));
    }
    if (lane == 0) s_w[warp] = n;
    __syncthreads();
    if (warp == 0) {  // publish, look back, publish the prefix
      int total = 0;
#pragma unroll
      for (int w = 0; w < kCWarps; ++w) total += s_w[w];
      int64_t excl;
      if (t == 0) {
        excl = *A.total_dst;
      } else {
        if (lane == 0) atomicExch(reinterpret_cast<unsigned long long*>(status + t), kFlagAgg | (uint64_t)total);
        excl = look_back(status, t, A.flags);
      }
      if (lane == 0) {
        atomicExch(reinterpret_cast<unsigned long long*>(status + t), kFlagPrefix | (uint64_t)(excl + total));
        s_base = excl;
        if (mark0 == 0 && A.event_offsets_out) A.event_offsets_out[A.ev_lo + row] = excl;
        if (t == n_t - 1) *A.total_dst = excl + total;
      }
    }
    __syncthreads();
    int64_t pos = s_base;
    for (int w = 0; w < warp; ++w) pos += s_w[w];
    for (int k = lo; k < hi; k += kLoads) {
      if (hi - lo > kLoads) load(k);
#pragma unroll
      for (int j = 0; j < kLoads; ++j) {
        const bool nx = acc_nonzero(v[j].x), ny = acc_nonzero(v[j].y);
        const unsigned mx = __ballot_sync(0xffffffffu, nx), my = __ballot_sync(0xffffffffu, ny);
        if (!(mx | my)) continue;
        const int group = s_list[k + j];
        if (nx || ny) cells[32 * group] = make_double2(0.0, 0.0);
        int64_t p = pos + __popc(mx & below) + __popc(my & below);
        const int c = (group << kMarkShift) + 2 * lane;
        const bool px = p < A.capacity && A.cell_ids, py = p + (nx ? 1 : 0) < A.capacity && A.cell_ids;
        if (nx && (DENSE || px)) {
          const float E = acc_to_f32(v[j].x);
          if (DENSE) dense[c] = E;
          if (px) {
            A.cell_ids[p] = c;
            A.cell_E[p] = E;
          }
        }
        p += nx ? 1 : 0;
        if (ny && (DENSE || py)) {
          const float E = acc_to_f32(v[j].y);
          if (DENSE) dense[c + 1] = E;
          if (py) {
            A.cell_ids[p] = c + 1;
            A.cell_E[p] = E;
          }
        }
        pos += __popc(mx) + __popc(my);
      }
    }
    __syncthreads();  // the shared arrays are reused
  }
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1ull) == (unsigned long long)gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int64_t i = tid; i < n_t; i += kCThreads) status[i] = 0;
    if (tid == 0) {
      *ticket = 0;
      *done = 0;
    }
  }
}

}  // namespace

cudaError_t launch_compact(const GeoDev& g, WsDev w, int32_t rows, int32_t ev_lo, ScanTmp tmp, float* cells_out,
                           int32_t* cell_ids, float* cell_E, int64_t* event_offsets_out, int64_t capacity, int max_ctas,
                           const Launch& L) {
  if (rows <= 0) return cudaSuccess;
  const int cpr = (g.n_cells + kChunk - 1) / kChunk;
  const int64_t n_chunks = (int64_t)rows * cpr;
  // persistent CTAs (the ticket order makes every look-back wait end); the
  // offsets continue the call's running output size (per-event mode)
  const int grid = (int)std::min<int64_t>(n_chunks, max_ctas > 0 ? max_ctas : (int64_t)L.num_sms * kCtasPerSm);
  const CompactArgs A{w.acc, g.n_cells, g.acc_stride, cpr, ev_lo, max_ctas > 0 ? 1 : 0, n_chunks, tmp.state, tmp.cap_tiles, tmp.flags,
                      &w.sizes->nnz_total, cells_out, cell_ids, cell_E, event_offsets_out, capacity};
  const auto kernel = cells_out && cell_ids ? k_compact_one<true, true>
                      : cells_out           ? k_compact_one<true, false>
                      : cell_ids            ? k_compact_one<false, true>
                                            : k_compact_one<false, false>;
  if (max_ctas > 0) {  // on a stream of its own, behind another stream's event
    kernel<<<grid, kCThreads, 0, L.s>>>(A);
    return cudaGetLastError();
  }
  return launch_dependent(kernel, grid, kCThreads, 0, L.s, A);
}

cudaError_t launch_compact_sparse(const GeoDev& g, WsDev w, int32_t rows, int32_t ev_lo, ScanTmp tmp, float* cells_out,
                                  int32_t* cell_ids, float* cell_E, int64_t* event_offsets_out, int64_t capacity,
                                  const Launch& L) {
  if (rows <= 0) return cudaSuccess;
  // (no more parts than the row has chunks: the scan state's size)
  const int parts = std::max(1, std::min((g.n_cells + kChunk - 1) / kChunk, kSparseParts / rows));
  const int64_t n_parts = (int64_t)rows * parts;
  const int grid = (int)std::min<int64_t>(n_parts, (int64_t)L.num_sms * kSparseCtas);
  const CompactArgs A{w.acc, g.n_cells, g.acc_stride, parts, ev_lo, 0, n_parts, tmp.state, tmp.cap_tiles, tmp.flags,
                      &w.sizes->nnz_total, cells_out, cell_ids, cell_E, event_offsets_out, capacity};
  return launch_dependent(cells_out ? k_compact_sparse<true> : k_compact_sparse<false>, grid, kCThreads, 0, L.s, A, w.marks);
}

int64_t compact_chunks(int32_t n_cells, int32_t rows) {
  return (int64_t)rows * ((n_cells + kChunk - 1) / kChunk);
}

}  // namespace fcs
