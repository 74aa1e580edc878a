// fcs_hits_impl.cuh - launch dispatch of the hit kernel over its block sizes; included by the atomic-mode,
// deterministic-mode and gradient-mode translation units.
#pragma once

#include "fcs_hits.cuh"

namespace fcs {

static inline HitKParams make_hit_params(const GeoDev& g, const ParamDev& p, WsDev w, int32_t ev_lo, uint32_t k0,
                                         uint32_t k1, int64_t first_event, int key_task_bits,
                                         const fcs_debug* dbg) {
  HitKParams kp{};
  kp.g = g;
  kp.p = p;
  kp.w = w;
  kp.ev_lo = ev_lo;
  kp.k0 = k0;
  kp.k1 = k1;
  kp.first_event_lo = (uint32_t)first_event;
  kp.key_task_bits = key_task_bits;
  kp.key32 = g.n_cells < (1 << 27) ? 1 : 0;
  kp.dbg_hit_cell = dbg ? dbg->hit_cell : nullptr;
  kp.dbg_hit_bin = dbg ? dbg->hit_bin : nullptr;
  kp.dbg_hit_cap = dbg ? dbg->hit_capacity : 0;
  kp.rk = philox_round_keys(k0, k1);
  return kp;
}

template <int BLOCK, int MODE, bool DBG, bool SPARSE = false>
static cudaError_t launch_hits_kernel(const HitKParams& kp, const Launch& L) {
  static int occ = -1;  // resident CTAs per SM of this instantiation
  if (occ < 0) {
    int o = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_hits<BLOCK, MODE, DBG, SPARSE>, BLOCK, 0);
    if (e != cudaSuccess) return e;
    occ = o < 1 ? 1 : o;
  }
  int64_t grid = (int64_t)L.num_sms * occ;
  if (kp.static_tiles) {
    const int64_t per_cta = (int64_t)kp.ticket * (BLOCK / 32);
    grid = (kp.h_hi - kp.h_lo + per_cta - 1) / per_cta;
    if (grid <= 0) return cudaSuccess;
  }
  return launch_dependent(k_hits<BLOCK, MODE, DBG, SPARSE>, grid, BLOCK, 0, L.s, kp);
}

// The validation dumps run in their own instantiation (no gradient-mode dumps).
template <int BLOCK, int MODE>
static cudaError_t launch_hits_block(const HitKParams& kp, const Launch& L) {
  if constexpr (MODE != kModeGrad) {
    if (kp.dbg_hit_cell || kp.dbg_hit_bin) return launch_hits_kernel<BLOCK, MODE, true>(kp, L);
  }
  if constexpr (MODE != kModeGrad) {
    if (kp.w.marks) return launch_hits_kernel<BLOCK, MODE, false, true>(kp, L);
  }
  return launch_hits_kernel<BLOCK, MODE, false>(kp, L);
}

// hc.hpt sets the queue's tickets, kGranule hits per unit (at most
// kMaxTicket); 0 leaves them to the kernel, which knows the call's hits.
template <int MODE>
cudaError_t launch_hits_t(const HitKParams& kp0, const HitCfg& hc, const Launch& L) {
  HitKParams kp = kp0;
  kp.ticket = std::min(hc.hpt * kGranule, kMaxTicket);
  if (kp.static_tiles && !kp.ticket) kp.ticket = 2 * kGranule;
  switch (hc.block) {
    case 128: return launch_hits_block<128, MODE>(kp, L);
    case 256: return launch_hits_block<256, MODE>(kp, L);
    case 512: return launch_hits_block<512, MODE>(kp, L);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE>
cudaError_t launch_recheck_t(const HitKParams& kp, const Launch& L) {
  // FP64 work: small blocks spread the queue over every SM's FP64 pipe
  return launch_dependent(k_recheck<MODE>, L.num_sms * 8, 64, 0, L.s, kp);
}

}  // namespace fcs
