// fcs_params.cu - builds the inverse-CDF thresholds and guide tables of the
// shape histograms on the device.
//
// Thresholds: with C_k the FP64 left-to-right prefix sum of the first k
// weights and K the last bin of non-zero weight, T[k] = min(2^32 - 1,
// floor(2^32 C_{k+1} / C_128)) for k < K and 2^32 - 1 for k >= K.  The bin of
// a 32-bit random word x is the first k < K with x < T[k], else K.
//
// Guide table (Chen and Asau's indexed search): for guide cell j (the words
// with x >> 24 == j) lo_j is the bin of x = j << 24 and hi_j the bin of
// x = (j + 1) << 24 (K for the last cell); the bin of every x in the cell lies
// in [lo_j, hi_j] and equals lo_j plus the number of thresholds T[k],
// lo_j <= k < hi_j, with T[k] <= x (T does not decrease).  Within the cell
// such a threshold satisfies j 2^24 < T[k] <= (j + 1) 2^24, so it is stored
// exactly as the 24-bit offset t_k = T[k] - j 2^24 - 1, and x >= T[k] reads
// (x mod 2^24) > t_k.  A cell packs, in 32 bits, t_lo (the value 2^24 - 1,
// which no offset exceeds, where the cell holds no threshold), lo_j and whether
// it holds more than one:
//   t_lo << 8 | lo_j << 1 | (hi_j - lo_j > 1),
// so that (x << 8) > cell is the comparison as it stands.  The bin of a word
// is decided by one 4-byte load and one comparison unless the cell holds two
// or more thresholds and x lies past the first (2 % of the words of the
// falling histograms); then a binary search over T[lo_j + 1 ..] finishes it.
// 256 cells of one threshold against 128 of two in 8 bytes: the same row of
// 1 KB and the same share of searches, half the instructions to decode.
#include "fcs_internal.cuh"

namespace fcs {
namespace {

constexpr uint32_t kGuideNever = 0xFFFFFFu;  // an offset no word of the cell exceeds

__device__ __forceinline__ uint32_t guide_cell(uint32_t t0, int lo, int span) {
  return (t0 << 8) | ((uint32_t)lo << 1) | (span > 1 ? 1u : 0u);
}

// The entries whose tables are to be built: those with a layer fraction > 0
// (no other entry has tasks, so no other table is read), all of them or those
// not built since the weights last changed.  built: per entry, whether its
// tables belong to the present weights.
__global__ void __launch_bounds__(256) k_table_list(const float* __restrict__ frac, int n_entries, int all,
                                                    uint8_t* __restrict__ built, int32_t* __restrict__ list,
                                                    int32_t* __restrict__ n_list) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  bool need = false;
  if (e < n_entries) {
    need = frac[e] > 0.0f && (all || !built[e]);
    if (need) built[e] = 1;
    else if (all) built[e] = 0;
  }
  const unsigned m = __ballot_sync(0xffffffffu, need);
  if (!m) return;
  int base = 0;
  if (lane == 0) base = atomicAdd(n_list, __popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (need) list[base + __popc(m & ((1u << lane) - 1u))] = e;
}

// Tables of the listed entries, 32 to a warp, one per lane: the prefix sums of
// an entry are one chain of FP64 additions in the order of the definition, so
// an entry is a lane's work, and the rows move through shared memory so that
// every global access is a whole row.  The warp's rows take the 128 weights of
// its 32 entries ([bin][lane]), then their thresholds in the same place, then
// 32 guide cells of each at a time.
//
// The quotient 2^32 c / C is not divided out: with R = 2^32 / C rounded once,
// c R is within 2^-52 2^32 = 2^-20 of the exact quotient and the rounded one
// within 2^-21 of it, so its floor is that of c R unless c R lies within 3 2^-20
// of an integer (one threshold in 2^18), where the division decides.  FP64
// instructions per weight: two additions and a product (a division alone is
// ten times that; the FP64 pipe takes one warp instruction in 16 cycles).
// 122,400 entries, 28 % of them with a fraction, in a training step's update:
// 0.64 ms for one thread per entry reading its own row and dividing, 0.75 ms
// with the 256-cell guide, 0.07 ms here (0.095 before the rows were loaded four at
// a time and the sweep kept the next thresholds in registers).
constexpr int kTableWarps = 2;
constexpr int kTableRow = 33;  // [bin][lane], padded for the row-wise accesses

__global__ void __launch_bounds__(32 * kTableWarps) k_build_tables(const float* __restrict__ shape_w,
                                                                   const int32_t* __restrict__ list,
                                                                   const int32_t* __restrict__ n_list,
                                                                   uint32_t* __restrict__ thr,
                                                                   uint32_t* __restrict__ guide) {
  __shared__ uint32_t s_rows[kTableWarps][kNBins * kTableRow];
  __shared__ uint32_t s_cells[kTableWarps][32 * kTableRow];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  uint32_t* rows = s_rows[wi];
  uint32_t* cells = s_cells[wi];
  const int n = *n_list;
  for (int g = (blockIdx.x * kTableWarps + wi) * 32; g < n; g += gridDim.x * kTableWarps * 32) {
    const int cnt = min(32, n - g);
    const int mine = list[g + min(lane, cnt - 1)];
    __syncwarp();
    // (rows past cnt are the last entry's again; four rows' loads in flight)
#pragma unroll 1
    for (int j0 = 0; j0 < 32; j0 += 4) {
      float v[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int e = __shfl_sync(0xffffffffu, mine, j0 + j);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[j][q] = __ldg(shape_w + (int64_t)e * kNBins + lane + 32 * q);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) rows[(lane + 32 * q) * kTableRow + j0 + j] = __float_as_uint(v[j][q]);
    }
    __syncwarp();
    double C = 0.0;
    int K = -1;
#pragma unroll 4
    for (int k = 0; k < kNBins; ++k) {
      const float w = __uint_as_float(rows[k * kTableRow + lane]);
      C = __dadd_rn(C, f32_to_f64_bits(w));
      if (w > 0.0f) K = k;
    }
    const bool good = C > 0.0 && K >= 0;  // the loaders' checks refuse the others
    const double R = good ? __ddiv_rn(4294967296.0, C) : 0.0;
    double c = 0.0;
#pragma unroll 4
    for (int k = 0; k < kNBins; ++k) {
      c = __dadd_rn(c, f32_to_f64_bits(__uint_as_float(rows[k * kTableRow + lane])));
      uint32_t T = 0xFFFFFFFFu;
      if (good && k < K) {
        // v = m 2^(e - 52), m the 53-bit significand: its floor and the 20
        // bits below the point by shifts
        const double v = __dmul_rn(c, R);
        const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
        const int ex = (int)(hi >> 20) - 1023;
        const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
        uint64_t fx = 0;  // v 2^20, truncated
        if (ex >= -20) fx = ex <= 32 ? m >> (32 - ex) : ~0ull;
        const uint32_t frac20 = (uint32_t)fx & 0xFFFFFu;
        uint64_t t = fx >> 20;
        if (frac20 <= 2u || frac20 >= 0xFFFFDu) {  // too near to an integer: the definition
          const double d = floor(__ddiv_rn(__dmul_rn(4294967296.0, c), C));
          t = d > 4294967295.0 ? 0xFFFFFFFFull : (uint64_t)d;
        }
        T = t > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)t;
      }
      rows[k * kTableRow + lane] = T;
    }
    __syncwarp();
#pragma unroll 4
    for (int j = 0; j < cnt; ++j) {
      const int e = __shfl_sync(0xffffffffu, mine, j);
#pragma unroll
      for (int q = 0; q < 4; ++q) thr[(int64_t)e * kNBins + lane + 32 * q] = rows[(lane + 32 * q) * kTableRow + j];
    }
    // lo_j = first k < K with (j << 24) < T[k], else K (monotone sweep); cell j
    // ends where the next begins, the last one at K
    // (Tk: the threshold k, and Tn the one after it, loaded ahead of its use)
    int k = 0;
    uint32_t Tk = rows[lane], Tn = rows[kTableRow + lane];
    auto step = [&]() {
      ++k;
      Tk = Tn;
      Tn = rows[min(k + 1, kNBins - 1) * kTableRow + lane];
    };
    while (k < K && Tk == 0u) step();  // lo_0: bins of zero weight before the first
    for (int j0 = 0; j0 < kGuideCells; j0 += 32) {
#pragma unroll 4
      for (int j = 0; j < 32; ++j) {
        const int lo = k;
        const uint32_t base = (uint32_t)(j0 + j) << 24;
        const uint32_t t0 = Tk;
        int span = 0;
        if (j0 + j + 1 < kGuideCells) {
          while (k < K && base + 0x1000000u >= Tk) {
            step();
            ++span;
          }
        } else {
          span = max(K, 0) - k;
        }
        cells[j * kTableRow + lane] = guide_cell(good && span >= 1 ? t0 - base - 1u : kGuideNever, good ? lo : 0,
                                                 good ? span : 0);
      }
      __syncwarp();
#pragma unroll 8
      for (int j = 0; j < cnt; ++j) {
        const int e = __shfl_sync(0xffffffffu, mine, j);
        guide[(int64_t)e * kGuideCells + j0 + lane] = cells[lane * kTableRow + j];
      }
      __syncwarp();
    }
  }
}

}  // namespace

cudaError_t launch_build_tables(const float* frac, const float* shape_w, int n_entries, int all, uint8_t* built,
                                int32_t* list, int32_t* n_list, uint32_t* thr, uint32_t* guide, cudaStream_t s) {
  if (n_entries <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(n_list, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  k_table_list<<<(n_entries + 255) / 256, 256, 0, s>>>(frac, n_entries, all, built, list, n_list);
  const int groups = (n_entries + 31) / 32;  // at most; a warp without a group ends at once
  k_build_tables<<<(groups + kTableWarps - 1) / kTableWarps, 32 * kTableWarps, 0, s>>>(shape_w, list, n_list, thr,
                                                                                      guide);
  return cudaGetLastError();
}

}  // namespace fcs
