// fcs_hits.cuh - the per-hit kernel of the hit loop (Listing 1: simulate_hit
// chain; Listing 2: HitCellMapping_d / getDDE + atomicAdd).
//
// One thread per hit as in the paper's sim_a kernel (Sec. 4), but persistent:
// CTAs take tiles of BLOCK * HPT consecutive hits from an atomic work queue
// over the whole batch (the grouped simulation of Sec. 4 at batch scale); a
// tile's tasks are staged in shared memory, each with its hits' map to scaled
// cell indices folded into one multiply-add per coordinate, and each hit finds
// its task by counting the task starts at or before it.  Per hit:
//   Philox4x32-10 block (hit, layer, particle, event)        -> 4 words
//   word 0: shape bin by guide table + binary search          (integer, exact)
//   words 1, 2: uniform position in the (r, alpha) bin        (FP32)
//   (r, alpha) -> scaled (eta, phi) cell indices of the task's home region
//     (FP32, __sincosf)
// The FP32 result is certified against a rigorous error bound.  A hit that
// leaves the home region or lies within the bound of a cell edge (about one in
// 200) takes the search over the layer's regions, certified likewise; what
// stays uncertain (one in 5000) is queued and decided by the FP64 recheck
// kernel, which repeats the oracle's FP64 steps (the paper's two FP32 cell
// mismatches in 62M hits were removed with FP64, Sec. 6).  Certified hits are
// deposited with warp-aggregated atomics (Sec. 4 chose atomicAdd) of the float
// count x Ehit into FP64 cells or, in deterministic mode, emitted as (cell,
// task, count) records for the sort-by-cell reduction.
#pragma once

#include "fcs_internal.cuh"

namespace fcs {

constexpr int kMaxTicket = 1024;  // hits a warp takes from the work queue at a time, at most

struct HitKParams {
  GeoDev g;
  ParamDev p;
  WsDev w;
  int32_t ev_lo;
  uint32_t k0, k1;
  uint32_t first_event_lo;
  int32_t key_task_bits;
  int32_t key32;  // 32-bit (cell, task in pass) match keys (n_cells < 2^27)
  int32_t* dbg_hit_cell;
  int16_t* dbg_hit_bin;
  int64_t dbg_hit_cap;
  // gradient mode
  const float* grad_in;  // dL/dE_cell of the range's events, row stride n_cells
  double* grad_acc;      // [n_entries][128] sum of E_hit dL/dE_cell per (entry, shape bin)
  uint8_t* grad_touched; // [n_entries] set where grad_acc has contributions
  int32_t ticket;        // hits per queue ticket, a multiple of kGranule up to kMaxTicket; 0: from the call's hits
  // one launch per task (static_tiles != 0): warp b of the grid takes tile b
  // of the hits [h_lo, h_hi), all of task t_last
  int64_t h_lo, h_hi;
  int32_t t_last;
  int32_t static_tiles;
  PhiloxRoundKeys rk;  // the round keys of (k0, k1), read from the parameter bank
};

// ---- shape bin: inverse CDF by guide table and binary search --------------
// The bin of word x0 for an entry whose bins below lo lie below x0: the first
// k >= lo with x0 < T[k].  T is 2^32 - 1 from the last bin K
// of non-zero weight on, so K is found for every word but 2^32 - 1, which is
// below no threshold and belongs to K.
static __device__ __noinline__ int bin_search(const ParamDev& p, uint32_t gbase, int lo, uint32_t x0) {
  if (x0 == 0xFFFFFFFFu) {
    int k = kNBins - 1;
    while (k > 0 && !(__ldg(p.shape_w + gbase + k) > 0.0f)) --k;
    return k;
  }
  // most searches end within four thresholds: they are loaded at once
  int n = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) n += x0 >= __ldg(p.thr + gbase + min(lo + j, kNBins - 1)) ? 1 : 0;
  lo += n;
  if (n < 4) return lo;
  int hi = kNBins - 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (x0 < __ldg(p.thr + gbase + mid)) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// The bin of word x0: the guide cell of x0's top 8 bits gives lo and the
// cell's first threshold as an offset (fcs_params.cu); one comparison decides
// unless the cell holds two or more thresholds and x0 lies past the first (two
// words in a hundred), which finishes with a binary search over the
// thresholds.  gbase: the entry x 128 (its first threshold; its first guide
// cell is 2 gbase).
struct GuideBin {
  int bin;      // the bin, or the first bin of the search
  bool search;
};
__device__ __forceinline__ uint32_t guide_word(const ParamDev& p, uint32_t gbase, uint32_t x0) {
  return __ldg(p.guide + (2u * gbase + (x0 >> 24)));
}
__device__ __forceinline__ GuideBin bin_in_cell(uint32_t x0, uint32_t g) {
  const bool past = (x0 << 8) > g;  // x0 past the threshold (the low byte of g does not reach the offset's bits)
  return {(int)((g >> 1) & 0x7Fu) + (past ? 1 : 0), past && (g & 1u)};
}
__device__ __forceinline__ int sample_bin(const ParamDev& p, uint32_t gbase, uint32_t x0) {
  const GuideBin b = bin_in_cell(x0, guide_word(p, gbase, x0));
  return b.search ? bin_search(p, gbase, b.bin, x0) : b.bin;
}

// ---- FP64 path: the oracle's steps, each rounding once ----------------------
__device__ __forceinline__ void scales64(const GeoDev& g, int layer, double eta_c, double* s_eta,
                                         double* s_phi) {
  const double R = g.rz[layer];
  if (g.barrel[layer]) {
    *s_phi = __ddiv_rn(1.0, R);
    *s_eta = __ddiv_rn(1.0, __dmul_rn(R, cosh(eta_c)));
  } else {
    const double ae = fabs(eta_c);
    const double sh = sinh(ae);
    const double m = __ddiv_rn(__dmul_rn(tanh(ae), sh), R);
    *s_phi = __ddiv_rn(sh, R);
    *s_eta = (eta_c < 0.0) ? m : -m;
  }
}

// The eta and phi indices in region r.
__device__ __forceinline__ int32_t eta_index64(const GeoDev& g, int r, double eta) {
  const int ne = g.n_eta[r];
  const double te = __ddiv_rn(__dsub_rn(eta, g.eta_lo[r]), g.deta[r]);
  if (!(te >= 0.0)) return 0;  // also NaN
  if (te >= (double)ne) return ne - 1;
  return min((int32_t)floor(te), ne - 1);  // te < n_eta <= 2^22
}
__device__ __forceinline__ int32_t phi_index64(const GeoDev& g, int r, double phi) {
  const int np = g.n_phi[r];
  double tp = __ddiv_rn(__dsub_rn(phi, g.phi_lo[r]), g.dphi[r]);
  const double lim = 4503599627370496.0;
  if (tp > lim) tp = lim;
  if (!(tp >= -lim)) tp = -lim;  // also NaN
  const double f = floor(tp);
  int32_t ip;
  if (fabs(f) < 2147483648.0) ip = (int32_t)f % np;
  else ip = (int32_t)((int64_t)f % (int64_t)np);
  return ip < 0 ? ip + np : ip;
}

__device__ __forceinline__ int32_t lookup64(const GeoDev& g, int layer, double eta, double phi) {
  const int rb = g.lrb[layer], re = g.lrb[layer + 1];
  int r = rb;
  for (int k = rb + 1; k < re; ++k)
    if (eta >= g.split[k]) r = k;
  return g.cell_off[r] + eta_index64(g, r, eta) * g.n_phi[r] + phi_index64(g, r, phi);
}

static __device__ __noinline__ int32_t cell_fp64(const GeoDev& g, const ParamDev& p, int32_t layer,
                                                 float eta_c, float phi_c, uint4 x, int bin) {
  const int ir = bin >> 3, ia = bin & 7;
  const double r_lo = (double)p.r_edges[ir], r_hi = (double)p.r_edges[ir + 1];
  const double a_lo = (double)p.a_edges[ia], a_hi = (double)p.a_edges[ia + 1];
  const double r = __dadd_rn(r_lo, __dmul_rn(u24d(x.y), __dsub_rn(r_hi, r_lo)));
  const double alpha = __dadd_rn(a_lo, __dmul_rn(u24d(x.z), __dsub_rn(a_hi, a_lo)));
  double s_eta, s_phi;
  scales64(g, layer, (double)eta_c, &s_eta, &s_phi);
  const double deta = __dmul_rn(__dmul_rn(r, cos(alpha)), s_eta);
  const double dphi = __dmul_rn(__dmul_rn(r, sin(alpha)), s_phi);
  const double eta = __dadd_rn((double)eta_c, deta);
  const double phi = __dadd_rn((double)phi_c, dphi);
  return lookup64(g, layer, eta, phi);
}

// ---- search over the layer's regions (FP32, certified) -------------------------
// For the hits that the staged map of the home region cannot certify.
// Error bound of the FP32 eta (and likewise phi) against the FP64 value:
//   cos/sin: |alpha32 - alpha| <= ~2^-21 (alpha - pi in [-pi, pi] from an
//     FMA of FP32 values) and __sincosf's documented absolute error on
//     [-pi, pi] (2^-21.19 for cos, 2^-21.41 for sin): <= 2^-20 in all;
//   r32 <= r_hi * 2^-23 off; s32 (coshf, sinhf and tanhf within 2, 3 and 2
//     ulp as documented, a correctly rounded 1/R or 1/cosh and up to two
//     products: <= 8 ulp) <= 2^-20 relative; the two products 2 * 2^-24
//     relative:
//   => |deta32 - deta| <= r_hi |s_eta| 2^-18.8; bound used: r_hi |s| 2^-17;
//   the final add rounds by |eta| 2^-24; bound used: |eta| 2^-21.
// Scaled index te = fl(eta32 inv + ek) with inv = fl(1/deta), ek =
// fl(-eta_lo/deta): |te - te*| <= be inv + (|eta| inv) 2^-24 + |ek| 2^-24 +
// |te| 2^-24 (the reciprocal, the constant and the FMA's rounding), and
// |eta| inv <= |te| + |ek|; bound used: be inv + |ek| 2^-23 + |te| 2^-21 +
// 2^-22; |ek| 2^-23 + 2^-22 is the region's constant ce (and likewise cp for
// phi).
// A decision is certified when the FP32 value is farther than the bound
// (plus the FP32 rounding of the boundary) from the boundary it is compared
// with.  Returns the cell, or -1 when a decision is not certified.
__device__ __forceinline__ int32_t generic_cell(const GeoDev& g, const ParamDev& p, const TaskRec& T, uint4 x,
                                                int bin) {
  const int ir = bin >> 3, ia = bin & 7;
  const float r_lo = __ldg(p.r_edges + ir), r_hi = __ldg(p.r_edges + ir + 1);
  const float a_lo = __ldg(p.a_edges + ia), a_hi = __ldg(p.a_edges + ia + 1);
  const float r = fmaf(u24f(x.y), r_hi - r_lo, r_lo);
  // alpha - pi (pi in two floats; within one more rounding of the FP64 difference)
  const float ap = fmaf(u24f(x.z), a_hi - a_lo, (a_lo - 3.14159274f) + 8.74227766e-8f);
  float sn, cs;
  __sincosf(ap, &sn, &cs);
  const float eta = T.eta_c + (r * -cs) * T.s_eta;
  const float phi = T.phi_c + (r * -sn) * T.s_phi;
  // the bounds r_hi |s| 2^-17 + |x| 2^-21 of the FP32 eta and phi
  const float be = fmaf(r_hi * 0x1p-17f, fabsf(T.s_eta), fabsf(eta) * 0x1p-21f);
  const float bp = fmaf(r_hi * 0x1p-17f, fabsf(T.s_phi), fabsf(phi) * 0x1p-21f);
  bool sure = fabsf(eta) < 1.0e30f;  // false for NaN or huge eta (a NaN phi fails its own test below)
  const int layer = T.layer(), rb = __ldg(g.lrb + layer), re = __ldg(g.lrb + layer + 1);
  int rr = rb;
  for (int q = rb + 1; q < re; ++q) {
    const float sp = __ldg(g.split32 + q);
    if (eta >= sp) rr = q;
    sure &= fabsf(eta - sp) > fmaf(fabsf(sp), 0x1p-23f, be);
  }
  const RegionF R = g.regf[rr];
  // eta index, clamped to [1/2, n_eta - 1/2]: outside it the cell is the first
  // or the last whichever side of the region's edge the hit lies, and at the
  // clamp the distance to the nearest integer is 1/2, so only interior cell
  // edges are certified
  const float te = fminf(fmaxf(fmaf(eta, R.inv_deta, R.ek), 0.5f), R.n_eta_hf);
  const float ke = rintf(te);
  sure &= fabsf(te - ke) > fmaf(te, 0x1p-21f, fmaf(be, R.inv_deta, R.ce));
  const int ie = (int)te;  // te >= 1/2: truncation is the floor
  const float tp = fmaf(phi, R.inv_dphi, R.pk);
  const float kp = rintf(tp);
  sure &= fabsf(tp - kp) > fmaf(fabsf(tp), 0x1p-21f, fmaf(bp, R.inv_dphi, R.cp));
  int ip = (int)floorf(tp) % R.n_phi;
  if (ip < 0) ip += R.n_phi;
  return sure ? R.cell_off + ie * R.n_phi + ip : -1;
}

// ---- staged tasks and the home region's map -----------------------------------
// The r and alpha bins as one multiply-add of f = 1 + u', f in [1, 2) built
// from the top 23 bits of a random word (u' = u without its last bit).
struct HitSmemTables {
  float2 rb[kNR];  // r = f rb.y + rb.x: lo - width, width
  float2 ab[kNA];  // alpha - pi = f ab.y + ab.x
};

__device__ __forceinline__ void load_tables(HitSmemTables& t, const ParamDev& p) {
  if (threadIdx.x < kNR) {
    const float lo = p.r_edges[threadIdx.x], hi = p.r_edges[threadIdx.x + 1];
    t.rb[threadIdx.x] = make_float2(lo - (hi - lo), hi - lo);
  }
  if (threadIdx.x < kNA) {
    const double lo = p.a_edges[threadIdx.x], hi = p.a_edges[threadIdx.x + 1];
    const float w = (float)(hi - lo);
    t.ab[threadIdx.x] = make_float2((float)(lo - 3.141592653589793 - (double)w), w);
  }
}

// A task as the hit loop uses it (80 B).  With inv = 1 / deta, ekh = -eta_lo /
// deta - 1/2 of the home region (and likewise phi), a hit's scaled index minus
// 1/2 is
//   te = (r cos(alpha - pi)) ea + eb,  ea = -s_eta inv,  eb = eta_c inv + ekh,
// one product and one multiply-add, and rint(te) is its cell index; pb is
// reduced by whole turns.  Bound of te's error, r eB + be + 1/2, with R the
// outer edge of the shape histogram:
//   r: u' is off by 2^-24; with the roundings of width, lo - width and the
//     FMA <= 5 2^-24 R;
//   alpha - pi: width w rounded (w - pi - lo formed with the rounded one),
//     u', the constant and the FMA's rounding: <= 2^-19.9 for any bin (2^-21.5
//     for the usual 8 bins); __sincosf 2^-21.19 absolute: <= 2^-19.4;
//   s32: <= 2^-20 relative (generic_cell); inv and the products 3 2^-24:
//   => r |ea| 2^-18.6 + R |ea| 5 2^-24; used: r |ea| 2^-17 + R |ea| 2^-21;
//   eb: (|eta_c| inv + |ekh| + |eb|) 2^-24 with |eta_c| inv <= |eb| + |ekh|,
//     and the FMA's rounding |te| 2^-24 <= n_eta 2^-24 wherever it decides
//     (beyond, te is clamped): used (|eb| + |ekh| + n_eta) 2^-23;
//   pb: likewise, and the reduction by whole turns rounds by n_phi 2^-23;
//   2^-21 absorbs second-order terms, the roundings of the bound itself and
//   neighbours' boundaries up to 2^-22 inside the grid (RegionF::fast_off).
// be and bp carry -1/2, so that a hit is certain when |te - rint(te)| <
// -(r eB + be), i.e. when its distance to the nearest cell edge exceeds the
// bound; a NaN or infinity anywhere fails the test.
struct __align__(16) TileTask {
  int32_t rel;      // first hit of the task - first hit of the pass (<= 0 for its first task)
  uint32_t gbase;   // parametrisation entry (with layer) x 128
  float Ehit;
  // Philox rounds 1 and 2 with the task's counter words folded in: only one
  // 32 x 32-bit product of each round depends on the hit
  uint32_t c0, c1, c2, c3;
  uint32_t base;    // accumulation row and region offset: + ie n_phi + ip, ie biased by kMagicBits
  int32_t n_phi;
  float ea, eb, pa, pb;
  float be, bp, eB, pB;
  float lo, hi;     // clamp of te (RegionF)
  float pad;
};
static_assert(sizeof(TileTask) == 80, "TileTask layout");

constexpr float kMagic = 12582912.0f;           // 1.5 2^23: adding it rounds to the nearest integer,
constexpr uint32_t kMagicBits = 0x4B400000u;    // which the low bits then hold (|x| < 2^22)

// The warp's view of task t: hit offset relative to the pass's first hit h0, the
// float hit energy fl32(El / n), the Philox counter words, the map and the
// accumulation row.
__device__ __forceinline__ TileTask make_tile_task(const WsDev& w, const GeoDev& g, int64_t t, int64_t h0,
                                                   uint32_t first_event_lo, int32_t ev_lo, uint32_t row_stride,
                                                   float r_max, const PhiloxRoundKeys& rk) {
  const TaskRec r = w.tasks[t];
  const RegionF R = g.regf[r.region()];
  const int32_t layer = r.layer(), event = r.event();
  TileTask q;
  q.rel = (int32_t)(w.th[t] - h0);
  q.gbase = (uint32_t)r.entry() * kNBins;
  q.Ehit = __fdiv_rn(r.El, (float)w.tn[t]);
  {  // counter (hit, layer | purpose << 16, particle in event, event): round 1's second product, round 2's first
    const uint32_t z = (uint32_t)r.particle;
    const uint32_t x1 = __umulhi(kPhiloxM1, z) ^ ((uint32_t)layer | (kPurposeHit << 16)) ^ rk.k[0];
    q.c0 = (first_event_lo + (uint32_t)event) ^ rk.k[1];
    q.c1 = kPhiloxM1 * z ^ rk.k[2];
    q.c2 = __umulhi(kPhiloxM0, x1) ^ rk.k[3];
    q.c3 = kPhiloxM0 * x1;
  }
  q.n_phi = R.n_phi;
  q.base = (uint32_t)(event - ev_lo) * row_stride + (uint32_t)R.fast_cell - kMagicBits * (uint32_t)R.n_phi;
  q.ea = -r.s_eta * R.inv_deta;
  q.eb = fmaf(r.eta_c, R.inv_deta, R.ekh);
  q.pa = -r.s_phi * R.inv_dphi;
  const float pb = fmaf(r.phi_c, R.inv_dphi, R.pkh);
  const float nf = (float)R.n_phi;
  q.pb = fmaf(-floorf(__fdividef(pb, nf)), nf, pb);
  q.eB = fabsf(q.ea) * 0x1p-17f;
  q.pB = fabsf(q.pa) * 0x1p-17f;
  q.be = fmaf(fabsf(q.eb) + fabsf(R.ekh) + R.n_eta, 0x1p-23f, fmaf(r_max * fabsf(q.ea), 0x1p-21f, 0x1p-21f)) +
         (R.fast_off - 0.5f);
  q.bp = fmaf(fabsf(pb) + fabsf(R.pkh) + 2.0f * nf, 0x1p-23f, fmaf(r_max * fabsf(q.pa), 0x1p-21f, 0x1p-21f)) - 0.5f;
  q.lo = R.lo;
  q.hi = R.hi;
  q.pad = 0.0f;
  return q;
}

// The hit's Philox block from the task's folded words: rounds 1 and 2, then
// the eight others.
__device__ __forceinline__ uint4 hit_block(const TileTask& T, uint32_t hit, const PhiloxRoundKeys& rk) {
  const uint32_t z1 = __umulhi(kPhiloxM0, hit) ^ T.c0, w1 = kPhiloxM0 * hit;
  uint4 c = make_uint4(__umulhi(kPhiloxM1, z1) ^ T.c1, kPhiloxM1 * z1, w1 ^ T.c2, T.c3);
#pragma unroll
  for (int i = 2; i < 10; ++i) c = philox_round(c, rk.k[2 * i], rk.k[2 * i + 1]);
  return c;
}

struct FastHit {
  uint32_t cell;  // accumulation row offset + cell
  bool sure;
};

__device__ __forceinline__ FastHit fast_cell(const HitSmemTables& tb, const TileTask& T, uint32_t x1, uint32_t x2,
                                              int bin) {
  const float2 rbin = tb.rb[bin >> 3], abin = tb.ab[bin & 7];
  // the top 23 bits of a word below the exponent of 1.0f
  const float r = fmaf(__uint_as_float(__funnelshift_r(x1, 0x7Fu, 9)), rbin.y, rbin.x);
  const float ap = fmaf(__uint_as_float(__funnelshift_r(x2, 0x7Fu, 9)), abin.y, abin.x);  // alpha - pi
  float sn, cs;
  __sincosf(ap, &sn, &cs);
  const float te = fminf(fmaxf(fmaf(r * cs, T.ea, T.eb), T.lo), T.hi);
  const float tp = fmaf(r * sn, T.pa, T.pb);
  const float ke = te + kMagic, kp = tp + kMagic;
  FastHit f;
  f.sure = fabsf(te - (ke - kMagic)) < -fmaf(r, T.eB, T.be) && fabsf(tp - (kp - kMagic)) < -fmaf(r, T.pB, T.bp);
  // the phi index wrapped into [0, n_phi): as unsigned numbers, the smaller of
  // ip and ip + n is ip + n exactly for ip < 0, that of ip and ip - n is ip - n
  // exactly for ip >= n (one turn either way; beyond, the search takes the hit)
  const uint32_t n = (uint32_t)T.n_phi;
  uint32_t ip = __float_as_uint(kp) - kMagicBits;
  ip = min(ip, ip + n);
  ip = min(ip, ip - n);
  f.sure = f.sure && ip < n;
  f.cell = T.base + __float_as_uint(ke) * n + ip;
  return f;
}

// ---- warp-level deposit / record emission -----------------------------------
// Deterministic mode: the first lane of each group (peers: its lanes) of equal
// (cell, task) keys in the warp writes the group's record (count - 1 in the low bits) and counts
// it in the cell's uint32 counter (the accumulation row).  A warp writes its
// records contiguously into chunks of kRecordChunk slots that it takes from
// the range's slot counter (a round that does not fit continues in the next
// chunk) and fills the rest of its last chunk with the empty record (all ones)
// when it ends, so the slots handed out hold every record and a few empty
// ones.  Uncertain hits are left to the recheck kernel.  Returns the warp's
// number of records (the caller counts them per CTA: one counter hit by every
// warp would serialise).
struct RecordChunk {
  int64_t base = 0;
  int fill = kRecordChunk;  // no chunk yet
};

template <bool SPARSE>
__device__ __forceinline__ unsigned emit_records(bool ok, unsigned peers, unsigned long long gkey, uint32_t cell,
                                                 RecordChunk& ch, const WsDev& w) {
  const int lane = threadIdx.x & 31;
  const bool lead = ok && (lane == __ffs(peers) - 1);
  const unsigned lm = __ballot_sync(0xffffffffu, lead);
  const int cnt = __popc(lm);
  if (cnt == 0) return 0u;
  const bool spill = ch.fill + cnt > kRecordChunk;
  unsigned long long nbase = 0;
  if (spill) {
    if (lane == 0) nbase = atomicAdd((unsigned long long*)&w.sizes->n_slots, (unsigned long long)kRecordChunk);
    nbase = __shfl_sync(0xffffffffu, nbase, 0);
  }
  if (lead) {
    const int pos = ch.fill + __popc(lm & ((1u << lane) - 1u));
    const int64_t slot = pos < kRecordChunk ? ch.base + pos : (int64_t)nbase + (pos - kRecordChunk);
    if (slot < w.rec_cap) {
      w.keys[slot] = (gkey << kRecordCountBits) | (unsigned long long)(__popc(peers) - 1);
      atomicAdd(reinterpret_cast<uint32_t*>(w.acc) + cell, 1u);
      if constexpr (SPARSE) set_mark(w.marks + (cell >> kMarkShift));
    } else {
      atomicOr(&w.sizes->flags, (uint32_t)FCS_FLAG_HIT_CAPACITY);
    }
  }
  if (spill) {
    ch.base = (int64_t)nbase;
    ch.fill += cnt - kRecordChunk;
  } else {
    ch.fill += cnt;
  }
  return (unsigned)cnt;
}

// The empty records after a warp's last one in its chunk.
__device__ __forceinline__ void close_records(const RecordChunk& ch, const WsDev& w) {
  for (int j = ch.fill + (threadIdx.x & 31); j < kRecordChunk; j += 32)
    if (ch.base + j < w.rec_cap) w.keys[ch.base + j] = ~0ull;
}

// A hit's E_hit dL/dE_cell, added in FP64 to the score of its (entry, bin).
// Each hit adds by itself: the 32 hits of a step fall into some 25 (entry, bin)
// pairs, so matching them first (2.2 cycles of the SM per distinct key) cost
// more than it saved (64 events, the whole backward call: 1348 to 1003 us).
__device__ __forceinline__ void grad_add(const HitKParams& kp, uint32_t key, float v) {
  atomicAdd(kp.grad_acc + key, (double)v);
}

__device__ __forceinline__ void deposit_single(const HitKParams& kp, int32_t event, float Ehit, int64_t task_rel,
                                               int32_t cell, int mode, int32_t entry, int bin) {
  const int64_t row = event - kp.ev_lo;
  if (mode == kModeAtomic) {
    acc_add(kp.w.acc + row * kp.g.acc_stride + cell, Ehit);
    if (kp.w.marks) set_mark(kp.w.marks + ((row * kp.g.acc_stride + cell) >> kMarkShift));
  } else if (mode == kModeGrad) {
    const float v = __fmul_rn(Ehit, __ldg(kp.grad_in + row * kp.g.n_cells + cell));
    atomicAdd(kp.grad_acc + ((int64_t)entry << 7) + bin, (double)v);
    kp.grad_touched[entry] = 1;
  } else {
    const uint32_t c = (uint32_t)(row * kp.g.acc_stride + cell);
    const unsigned long long gkey = ((unsigned long long)c << kp.key_task_bits) | (unsigned long long)task_rel;
    const int64_t slot = (int64_t)atomicAdd((unsigned long long*)&kp.w.sizes->n_slots, 1ull);  // a slot of its own
    if (slot < kp.w.rec_cap) {
      atomicAdd((unsigned long long*)&kp.w.sizes->n_records, 1ull);
      kp.w.keys[slot] = gkey << kRecordCountBits;
      atomicAdd(reinterpret_cast<uint32_t*>(kp.w.acc) + c, 1u);
      if (kp.w.marks) set_mark(kp.w.marks + (c >> kMarkShift));
    } else {
      atomicOr(&kp.w.sizes->flags, (uint32_t)FCS_FLAG_HIT_CAPACITY);
    }
  }
}

// The hits a warp has put off (one per lane, `have`: this lane has one): those
// whose bin needs the search over the thresholds and those the staged map did
// not certify.  Their cell comes from the search over the layer's regions, and
// where that is not certain either the hit is queued for the FP64 recheck
// kernel as (task, hit in task); when the queue is full its cell is decided
// here in FP64, as the recheck kernel would.  Called by the whole warp; out of
// line, as it runs once in some 50 warp steps (2 % of the hits, 32 at a time).
template <int MODE, bool DBG>
static __device__ __noinline__ void deferred_hits(const HitKParams& kp, bool have, uint2 th) {
  const WsDev& w = kp.w;
  TaskRec T{};
  uint4 x = make_uint4(0u, 0u, 0u, 0u);
  int bin = 0;
  int32_t c = -1;
  if (have) {
    T = w.tasks[th.x];
    x = philox4x32_10_rk(make_uint4(th.y, (uint32_t)T.layer() | (kPurposeHit << 16), (uint32_t)T.particle,
                                    kp.first_event_lo + (uint32_t)T.event()),
                         kp.rk);
    bin = sample_bin(kp.p, (uint32_t)T.entry() * kNBins, x.x);
    c = generic_cell(kp.g, kp.p, T, x, bin);
    if (c < 0) {
      const unsigned long long pos = atomicAdd((unsigned long long*)&w.sizes->n_recheck, 1ull);
      if (pos < (unsigned long long)w.recheck_cap) {
        w.recheck[pos] = th;
      } else {
        c = cell_fp64(kp.g, kp.p, T.layer(), T.eta_c, T.phi_c, x, bin);
        atomicAdd((unsigned long long*)&w.sizes->n_inline, 1ull);
        atomicOr(&w.sizes->flags, (uint32_t)FCS_FLAG_RECHECK_SPILL);
      }
    }
    if constexpr (DBG) {
      const int64_t h = w.sizes->hit_base + w.th[th.x] + th.y;
      if (h < kp.dbg_hit_cap) {
        if (kp.dbg_hit_cell && c >= 0) kp.dbg_hit_cell[h] = c;
        if (kp.dbg_hit_bin) kp.dbg_hit_bin[h] = (int16_t)bin;
      }
    }
  }
  const bool ok = c >= 0;
  const int64_t row = T.event() - kp.ev_lo;
  const float Ehit = ok ? __fdiv_rn(T.El, (float)w.tn[th.x]) : 0.0f;
  if constexpr (MODE == kModeGrad) {
    if (ok)
      grad_add(kp, ((uint32_t)T.entry() << 7) | (uint32_t)bin,
               __fmul_rn(Ehit, __ldg(kp.grad_in + row * kp.g.n_cells + c)));
  } else if constexpr (MODE == kModeAtomic) {
    if (ok) {
      acc_add(w.acc + row * kp.g.acc_stride + c, Ehit);
      if (w.marks) set_mark(w.marks + ((row * kp.g.acc_stride + c) >> kMarkShift));
    }
  } else {
    // records as emit_records writes them, in slots of their own
    const int lane = threadIdx.x & 31;
    const uint32_t cg = (uint32_t)(row * kp.g.acc_stride + c);
    const unsigned long long gkey = ((unsigned long long)cg << kp.key_task_bits) | th.x;
    const unsigned peers = __ballot_sync(0xffffffffu, ok) & __match_any_sync(0xffffffffu, gkey);
    const bool lead = ok && lane == __ffs(peers) - 1;
    const unsigned lm = __ballot_sync(0xffffffffu, lead);
    unsigned long long base = 0;
    if (lane == 0 && lm) {
      base = atomicAdd((unsigned long long*)&w.sizes->n_slots, (unsigned long long)__popc(lm));
      atomicAdd((unsigned long long*)&w.sizes->n_records, (unsigned long long)__popc(lm));
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    if (lead) {
      const int64_t slot = (int64_t)base + __popc(lm & ((1u << lane) - 1u));
      if (slot < w.rec_cap) {
        w.keys[slot] = (gkey << kRecordCountBits) | (unsigned long long)(__popc(peers) - 1);
        atomicAdd(reinterpret_cast<uint32_t*>(w.acc) + cg, 1u);
        if (w.marks) set_mark(w.marks + (cg >> kMarkShift));
      } else {
        atomicOr(&w.sizes->flags, (uint32_t)FCS_FLAG_HIT_CAPACITY);
      }
    }
  }
}

// Every warp works by itself: it takes a ticket of consecutive hits and runs
// through it in passes of up to NT tasks, one lane staging each, and the
// pass's hits 32 at a time, two steps in flight.  No warp waits for another:
// the long chains of dependent loads (a pass's task records, the hits put off)
// stall one warp and the others of the SM fill in.
//
// What bounds it: instruction issue, at 0.6-0.7 of the slots, behind the
// latency of the guide words (L2) that each step needs after its Philox block.
// 64 pile-up events (86.8M hits), this kernel's time on the library's events:
//   817 us  CTA tiles of 1024 hits with barriers, region tables in shared
//           memory, a search of the thresholds and the regions in the loop
//   768     one multiply-add per coordinate from staged tasks (1.7 fewer
//           conversions and table loads per hit), task starts as bits
//   729     neighbouring regions of one grid staged as one: 0.1 instead of
//           0.5 % of the hits leave the map
//   690     one 4-byte guide word, searches and uncertified hits put off to
//           full warps (in the loop their branches took half the steps)
//   598     a warp's own tickets and passes instead of CTA tiles
//   571     two steps in flight; 9 CTAs of 128 threads per SM at 56 registers
//           (10 at 48: 596, 8 at 64: 571, one step in flight: 600)
// SPARSE: the deposits set w.marks.
// (Finishing the searches in the loop with two more loads: 610.  Without any
// put-off hit, wrongly, it would be 500.)
//
// 9 CTAs of 128 threads per SM in every mode (of 7 to 10 tried).  DBG: the validation dumps of
// fcs_debug (a separate instantiation, so that the production kernel carries
// none of their code).
constexpr int hits_min_ctas(int block) { return 9 * 128 / block; }
template <int BLOCK, int MODE, bool DBG, bool SPARSE>
__global__ void __launch_bounds__(BLOCK, hits_min_ctas(BLOCK)) k_hits(const __grid_constant__ HitKParams kp) {
  dependent_start();
  constexpr bool DET = MODE == kModeDet;
  constexpr int NW = BLOCK / 32;
  constexpr int NT = BLOCK > 256 ? 24 : 32;  // staged tasks per warp (static shared memory holds 48 KB)
  constexpr unsigned kAll = 0xffffffffu;
  static_assert(kGuideCells == 2 * kNBins, "one base for guide cells and thresholds");
  static_assert(kMaxTicket <= 1024, "a pass's task starts are 32 words, one per lane");
  __shared__ HitSmemTables tb;
  __shared__ __align__(16) TileTask s_task[NW][NT];
  __shared__ uint32_t s_start[NW][32];  // bit i of the pass: a task other than its first starts at hit i
  __shared__ uint2 s_def[NW][96];       // hits put off (task, hit), fewer than 32 between rounds of two steps
  __shared__ unsigned long long s_recs;  // deterministic mode: records of this CTA
  load_tables(tb, kp.p);
  if (DET && threadIdx.x == 0) s_recs = 0;
  __syncthreads();
  const WsDev& w = kp.w;
  const int64_t H = kp.static_tiles ? kp.h_hi : w.sizes->n_hits;
  const int32_t T_end = kp.static_tiles ? kp.t_last + 1 : (int32_t)w.sizes->n_tasks;
  const int64_t hbase = kp.static_tiles ? kp.h_lo : 0;
  if (H > w.gmap_cap * (int64_t)kGranule) {  // the tile map is too small for the hits
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&w.sizes->flags, (uint32_t)FCS_FLAG_HIT_CAPACITY);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lanes_below = (1u << lane) - 1u, lanes_upto = lanes_below | (1u << lane);
  // Hits per ticket: as many as leave each warp several tickets, since a pass
  // of tasks costs as much as eight steps; small calls give each warp one.
  const uint32_t n_warps = gridDim.x * NW;
  const int64_t share = (H - hbase + n_warps - 1) / n_warps;  // hits per warp
  uint32_t q = (uint32_t)kp.ticket;
  if (q == 0) q = share > 4096 ? 1024u : share > 2048 ? 512u : share > 768 ? 256u : share > 256 || share <= 128 ? 128u : 256u;
  const uint32_t n_tiles = (uint32_t)((H - hbase + q - 1) / q);  // < 2^32: hits < 2^39
  // accumulation rows (atomic, deterministic) or dL/dE_cell rows (gradient)
  const uint32_t row_stride = MODE == kModeGrad ? (uint32_t)kp.g.n_cells : (uint32_t)kp.g.acc_stride;
  const float r_max = __ldg(kp.p.r_edges + kNR);
  unsigned long long recs = 0;  // deterministic mode: this warp's records
  RecordChunk chunk;            //   and the slots it writes them to
  int n_def = 0;                // this warp's hits in s_def
  // The first two thirds of the tickets go to the warps in turn, the rest
  // through the queue (its counter serves a ticket in 2.2 ns), which evens out
  // the warps' speeds; calls of many tickets a warp take all from the queue,
  // whose stricter order keeps the rows and tables in flight few (64 events:
  // 573 against 606 us; 7 events: 69 against 62 us).
  const uint32_t n_turns = kp.static_tiles ? 1u : share > 8192 ? 0u : max(n_tiles / n_warps * 2u / 3u, 1u);
  auto take = [&](uint32_t turn) {
    uint32_t t = turn * n_warps + blockIdx.x * NW + warp;
    if (turn >= n_turns) {
      t = n_tiles;
      if (!kp.static_tiles && lane == 0) t = n_turns * n_warps + (uint32_t)atomicAdd(&w.sizes->queue, 1ull);
    }
    return t;  // of the lane 0
  };
  uint32_t turn = 0;
  uint32_t tile = __shfl_sync(kAll, take(turn), 0);
  while (tile < n_tiles) {
    const uint32_t next = take(++turn);  // in flight during this ticket
    int64_t h0 = hbase + (int64_t)tile * q;  // first hit of the pass
    const int64_t h1 = min(h0 + (int64_t)q, H);
    int32_t t0 = kp.static_tiles ? kp.t_last : w.gmap[h0 / kGranule];
    while (h0 < h1) {
      // stage the tasks t0 .. t0 + NT - 1 and mark where each starts
      // (deterministic mode: the pass that holds a task's first hit writes the
      // task's hit energy for the fold)
      __syncwarp();
      s_start[warp][lane] = 0;
      __syncwarp();
      int end = (int)(h1 - h0);  // hits of the pass
      int after = end;           // where the lane's task ends
      if (lane < NT && t0 + lane < T_end) {
        const int64_t s64 = w.th[t0 + lane] - h0;
        if (s64 < end) {
          const TileTask t = make_tile_task(w, kp.g, t0 + lane, h0, kp.first_event_lo, kp.ev_lo, row_stride, r_max, kp.rk);
          s_task[warp][lane] = t;
          if (lane > 0) atomicOr(&s_start[warp][t.rel >> 5], 1u << (t.rel & 31));
          if (lane == NT - 1) after = (int)min((int64_t)end, s64 + w.tn[t0 + lane]);
          if constexpr (DET) {
            if (t.rel >= 0) w.tehit[t0 + lane] = t.Ehit;
          }
          if constexpr (MODE == kModeGrad) kp.grad_touched[t.gbase / kNBins] = 1;  // the task has hits
        }
      }
      end = __shfl_sync(kAll, after, NT - 1);
      __syncwarp();
      const uint32_t my_starts = s_start[warp][lane];
      int tbase = 0;  // tasks that start in the steps before
      // a step is 32 hits; its draw (task, random block, guide word) and its
      // finish (bin, cell, deposit) are apart so that a second step's load is
      // in flight before the first one's is used
      struct Draw {
        uint32_t x0, x1, x2, g, hit;
        int tl;
      };
      auto draw = [&](int k) {
        Draw d;
        const uint32_t starts = __shfl_sync(kAll, my_starts, k);
        d.tl = tbase + __popc(starts & lanes_upto);
        tbase += __popc(starts);
        const TileTask& T = s_task[warp][d.tl];
        d.hit = (uint32_t)(k * 32 + lane - T.rel);
        const uint4 x = hit_block(T, d.hit, kp.rk);
        d.x0 = x.x;
        d.x1 = x.y;
        d.x2 = x.z;
        d.g = guide_word(kp.p, T.gbase, x.x);
        return d;
      };
      auto finish = [&](int k, const Draw& d) {
        const TileTask& T = s_task[warp][d.tl];
        const GuideBin gb = bin_in_cell(d.x0, d.g);
        const int bin = gb.bin;
        const FastHit f = fast_cell(tb, T, d.x1, d.x2, bin);
        const bool valid = k * 32 + lane < end;
        const bool ok = valid && f.sure && !gb.search;
        if constexpr (MODE == kModeGrad) {
          // dL/dE_cell of the hit's cell times its energy, summed per (entry, bin)
          if (ok) grad_add(kp, T.gbase | (uint32_t)bin, __fmul_rn(T.Ehit, __ldg(kp.grad_in + f.cell)));
        } else {
          // the low 27 bits of the row offset + cell tell a task's cells apart
          // (n_cells < 2^27): with the task in the pass they identify (address, hit energy)
          const unsigned m = __ballot_sync(kAll, ok);
          const unsigned peers =
              m & (kp.key32 ? __match_any_sync(kAll, (f.cell << 5) | (uint32_t)d.tl)
                            : __match_any_sync(kAll, ((unsigned long long)(uint32_t)d.tl << 32) | f.cell));
          if constexpr (!DET) {
            if (ok && (peers & lanes_below) == 0u) {  // the group's first lane deposits
              acc_add(w.acc + f.cell, __fmul_rn((float)__popc(peers), T.Ehit));
              if constexpr (SPARSE) set_mark(w.marks + (f.cell >> kMarkShift));
            }
          } else {
            const unsigned long long gkey =
                ((unsigned long long)f.cell << kp.key_task_bits) | (unsigned long long)(t0 + d.tl);
            recs += emit_records<SPARSE>(ok, peers, gkey, f.cell, chunk, w);
          }
        }
        if constexpr (DBG) {
          const int64_t h = w.sizes->hit_base + h0 + k * 32 + lane;
          if (ok && h < kp.dbg_hit_cap) {
            if (kp.dbg_hit_cell)
              kp.dbg_hit_cell[h] =
                  (int32_t)(f.cell - (uint32_t)(w.tasks[t0 + d.tl].event() - kp.ev_lo) * row_stride);
            if (kp.dbg_hit_bin) kp.dbg_hit_bin[h] = (int16_t)bin;
          }
        }
        const unsigned md = __ballot_sync(kAll, valid && !ok);
        if (md) {  // put off
          if ((md >> lane) & 1u)
            s_def[warp][n_def + __popc(md & lanes_below)] = make_uint2((uint32_t)(t0 + d.tl), d.hit);
          n_def += __popc(md);
        }
      };
#pragma unroll 1
      for (int k = 0; k * 32 < end; k += 2) {
        const Draw d0 = draw(k);
        if ((k + 1) * 32 < end) {
          const Draw d1 = draw(k + 1);
          finish(k, d0);
          finish(k + 1, d1);
        } else {
          finish(k, d0);
        }
        if (n_def >= 32) {  // 32 put-off hits go through the search
          __syncwarp();
          do {
            n_def -= 32;
            deferred_hits<MODE, DBG>(kp, true, s_def[warp][n_def + lane]);
          } while (n_def >= 32);
          __syncwarp();
        }
      }
      h0 += end;
      t0 += NT;
    }
    tile = __shfl_sync(kAll, next, 0);
  }
  __syncwarp();
  if (n_def) deferred_hits<MODE, DBG>(kp, lane < n_def, s_def[warp][lane]);
  if constexpr (DET) {
    close_records(chunk, w);
    if (lane == 0 && recs) atomicAdd(&s_recs, recs);
    __syncthreads();
    if (threadIdx.x == 0 && s_recs) atomicAdd((unsigned long long*)&w.sizes->n_records, s_recs);
  }
}

// FP64 recheck of the queued hits, 32 to a block of two warps (grid-stride over
// the queue).
//
// Bound by latency: a dependent FP64 instruction takes 64 cycles, a division
// 560, sincos 1750, and a hit's map and lookup are one chain of them, whatever
// the queue's length.  So the two warps share a hit: the first holds the phi
// side (sine and cosine, the phi scale and index), the second the eta side (the
// hyperbolic functions, the eta scale, the region and the eta index), and what
// one needs of the other goes through shared memory.  cosh and sinh come from
// one exponential and its reciprocal (within 2 ulp of cosh's value and of
// sinh's absolute error, both below the rounding of the positions they move),
// and tanh sinh = sinh^2 / cosh.  Queues of up to some 30,000 hits: 12 to 16 us
// by one thread a hit and the functions one after the other; 9 to 12 us here (cold).
struct RecheckShared {
  double sn[32], cs[32];  // of alpha, by the first warp
  double sh[32];          // sinh |eta_c|, by the second
  double s_phi[32];       // |eta_c| > 20: the phi scale, by the second
  int region[32], ip[32];
};

template <int MODE>
__global__ void __launch_bounds__(64) k_recheck(const __grid_constant__ HitKParams kp) {
  dependent_start();
  __shared__ RecheckShared sm;
  const WsDev& w = kp.w;
  const GeoDev& g = kp.g;
  const int64_t n = min(w.sizes->n_recheck, w.recheck_cap);
  const int64_t hit_dbg_base = kp.dbg_hit_cell ? w.sizes->hit_base : 0;
  const int lane = threadIdx.x & 31;
  const bool eta_side = threadIdx.x >= 32;
  for (int64_t i0 = (int64_t)blockIdx.x * 32; i0 < n; i0 += (int64_t)gridDim.x * 32) {
    const int64_t i = i0 + lane;
    const bool have = i < n;
    const uint2 q = w.recheck[have ? i : i0];
    const TaskRec T = w.tasks[q.x];
    const int32_t layer = T.layer(), event = T.event();
    const uint4 x = philox4x32_10(
        make_uint4(q.y, (uint32_t)layer | (kPurposeHit << 16), (uint32_t)T.particle, kp.first_event_lo + (uint32_t)event),
        kp.k0, kp.k1);
    const int bin = sample_bin(kp.p, (uint32_t)T.entry() * kNBins, x.x);
    const int ir = bin >> 3, ia = bin & 7;
    const double r_lo = (double)kp.p.r_edges[ir], r_hi = (double)kp.p.r_edges[ir + 1];
    const double r = __dadd_rn(r_lo, __dmul_rn(u24d(x.y), __dsub_rn(r_hi, r_lo)));
    const double R = g.rz[layer];
    const bool barrel = g.barrel[layer] != 0;
    const int rb = g.lrb[layer], re = g.lrb[layer + 1];
    const double ec = (double)T.eta_c, ae = fabs(ec);
    const bool far = ae > 20.0;  // (sinh^2 overflows at 355; the functions themselves saturate)
    double sh = 0.0, ch = 0.0, s_eta = 0.0, s_phi = 0.0;
    if (eta_side) {
      const double e = exp(ae), ei = __ddiv_rn(1.0, e);
      ch = __dmul_rn(0.5, __dadd_rn(e, ei));
      sh = __dmul_rn(0.5, __dsub_rn(e, ei));
      if (far) scales64(g, layer, ec, &s_eta, &s_phi);
      sm.sh[lane] = sh;
      sm.s_phi[lane] = s_phi;
    } else {
      const double a_lo = (double)kp.p.a_edges[ia], a_hi = (double)kp.p.a_edges[ia + 1];
      const double alpha = __dadd_rn(a_lo, __dmul_rn(u24d(x.z), __dsub_rn(a_hi, a_lo)));
      double sn, cs;
      sincos(alpha, &sn, &cs);
      sm.sn[lane] = sn;
      sm.cs[lane] = cs;
    }
    __syncthreads();
    double pos;  // eta or phi of the hit
    int rr = rb;
    if (eta_side) {
      if (!far) {
        const double m = __ddiv_rn(barrel ? 1.0 : __dmul_rn(sh, sh), __dmul_rn(R, ch));
        s_eta = barrel || ec < 0.0 ? m : -m;
      }
      pos = __dadd_rn(ec, __dmul_rn(__dmul_rn(r, sm.cs[lane]), s_eta));
      for (int k = rb + 1; k < re; ++k)
        if (pos >= g.split[k]) rr = k;
      sm.region[lane] = rr;
    } else {
      s_phi = far ? sm.s_phi[lane] : __ddiv_rn(barrel ? 1.0 : sm.sh[lane], R);
      pos = __dadd_rn((double)T.phi_c, __dmul_rn(__dmul_rn(r, sm.sn[lane]), s_phi));
    }
    __syncthreads();
    rr = sm.region[lane];
    int32_t ie = 0;
    if (eta_side) {
      ie = eta_index64(g, rr, pos);
    } else {
      sm.ip[lane] = phi_index64(g, rr, pos);
    }
    __syncthreads();
    if (eta_side && have) {
      const int32_t c = g.cell_off[rr] + ie * g.n_phi[rr] + sm.ip[lane];
      deposit_single(kp, event, __fdiv_rn(T.El, (float)w.tn[q.x]), q.x, c, MODE, T.entry(), bin);
      const int64_t h = hit_dbg_base + w.th[q.x] + q.y;
      if (kp.dbg_hit_cell && h < kp.dbg_hit_cap) kp.dbg_hit_cell[h] = c;
    }
    // (the next round's first writes are to sn, cs, sh and s_phi, read before the last barrier)
  }
}

template <int MODE>
cudaError_t launch_hits_t(const HitKParams& kp, const HitCfg& hc, const Launch& L);

}  // namespace fcs
