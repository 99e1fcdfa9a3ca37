// Launch logic of the radix-16 team passes, instantiated per line length (team_<L>.cu).
#pragma once
#include <cuda_runtime.h>

#include "internal.h"
#include "team_pass.cuh"
#include "team_unsplit.cuh"

namespace dgb {

// As many CTAs as can be resident (128 registers: 512 threads per SM; each CTA takes its share
// of the tensor memory), at most one per work unit. The CTAs per SM follow from TGeo, as the
// occupancy query reports one CTA per SM for kernels that allocate tensor memory.
template <typename G, typename K, typename... A>
static cudaError_t launch_groups(K kern, bool (&configured)[64], int units, cudaStream_t st,
                                 A&&... args) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev]) {  // per kernel and device
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const int ctas = (units + G::GROUPS - 1) / G::GROUPS, most = G::MINB * sm_count();
  return launch_pdl(kern, dim3(ctas < most ? ctas : most), dim3(G::THREADS), G::SMEM, st, true, 0,
                    args...);
}

template <int L, int LPC, bool PAIR, bool BATCH, int SIGMA, int OUT>
static cudaError_t launch_team_as(const LinePassArgs<float>& a, cudaStream_t st) {
  using G = TGeo<L, LPC, PAIR>;
  if (a.n_lines % G::LPU != 0) return cudaErrorInvalidValue;
  static bool configured[64] = {false};
  const int units = (BATCH ? a.inst_capacity : 1) * (a.n_lines / G::LPU);
  return launch_groups<G>(line_pass_team<L, LPC, PAIR, BATCH, SIGMA, OUT>, configured, units, st, a,
                          units, a.err);
}

// How the lines are spread, by the points of a launch (all instances together):
//  up to 2^18  small CTAs (512 points at once), as many as possible: latency decides;
//  up to 2^20  CTAs of 2048 points, output staged in segments of 2048 / L lines;
//  above       pairs of lines per team, whole 32-byte sectors written from registers without
//              staging (batches from 2^21: their capacity, which sizes the launch, exceeds the
//              number of running instances by up to 2).
// Measured per step of two passes (ms), small | staged | pairs: 256^2 0.0109 | 0.0160 | 0.0239,
// 512 x 256 0.0121 | 0.0158, 512^2 0.0149 | 0.0154 | 0.0240, 1024 x 256 0.0153 | 0.0172 |
// 0.0257, 512 x 1024 0.0249 | 0.0193, 1024^2 - | 0.0325 | 0.0291, 512 x 2048 - | 0.0361 |
// 0.0301, 2048^2 - | 0.138 | 0.085.
template <int L, bool BATCH, int SIGMA, int OUT>
static cudaError_t launch_team_sized(const LinePassArgs<float>& a, cudaStream_t st) {
  constexpr int SMALL = L >= 512 ? 1 : 512 / L, LPC = L >= 2048 ? 1 : 2048 / L;
  const size_t points = (size_t)(BATCH ? a.inst_capacity : 1) * a.n_lines * L;
  if (points >= (BATCH ? kTeamPairPointsBatch : kTeamPairPoints))
    return launch_team_as<L, LPC, true, BATCH, SIGMA, OUT>(a, st);
  if (points <= ((size_t)1 << 18)) return launch_team_as<L, SMALL, false, BATCH, SIGMA, OUT>(a, st);
  return launch_team_as<L, LPC, false, BATCH, SIGMA, OUT>(a, st);
}

// The combinations the schemes use: sigma_x passes store transposed without U or rows with any
// (the symmetric order's last pass), sigma_y passes store transposed with any.
template <int L>
cudaError_t launch_team(const LinePassArgs<float>& a0, cudaStream_t st) {
  LinePassArgs<float> a = a0;
  if (!a.err || !a.tw_team || a.beta_im) return cudaErrorInvalidValue;
  a.tw = a.tw_team;
  if (a.inst) {
    if (a.store_normal || !a.n_inst) return cudaErrorInvalidValue;
    return a.sigma == 0 ? launch_team_sized<L, true, 0, TEAM_PLAIN>(a, st)
                        : launch_team_sized<L, true, 1, TEAM_U>(a, st);
  }
  if (!a.mult_perm || !a.beta || (a.u_store && a.ug_store)) return cudaErrorInvalidValue;
  if (a.sigma == 0) {
    if (a.store_normal)
      return a.u_load ? cudaErrorInvalidValue : launch_team_sized<L, false, 0, TEAM_ROWS>(a, st);
    if (a.u_store || a.ug_store) return cudaErrorInvalidValue;
    return launch_team_sized<L, false, 0, TEAM_PLAIN>(a, st);
  }
  if (a.store_normal || a.u_load) return cudaErrorInvalidValue;
  if (a.ug_store) return launch_team_sized<L, false, 1, TEAM_UG>(a, st);
  if (a.u_store) return launch_team_sized<L, false, 1, TEAM_U>(a, st);
  return launch_team_sized<L, false, 1, TEAM_PLAIN>(a, st);
}

template <int L, int LPC, bool PAIR, int PHASE>
static cudaError_t launch_unsplit_as(const UnsplitArgs& a, cudaStream_t st) {
  using G = TGeo<L, LPC, PAIR>;
  if (!a.in || !a.out || !a.beta || !a.tw || !a.mult || !a.err || a.n_lines % G::LPU != 0 ||
      (PHASE == 1 && !a.out_in) || (PHASE == 2 && !a.s_other))
    return cudaErrorInvalidValue;
  static bool configured[64] = {false};
  const int units = a.n_lines / G::LPU;
  return launch_groups<G>(line_pass_team_unsplit<L, LPC, PAIR, PHASE>, configured, units, st, a,
                          units);
}

// Pairs of lines from 2^20 points, as for the step pass.
template <int L>
cudaError_t launch_team_unsplit(const UnsplitArgs& a, int phase, cudaStream_t st) {
  constexpr int LPC = L >= 2048 ? 1 : 2048 / L;
  if ((size_t)a.n_lines * L >= kTeamPairPoints)
    return phase == 1 ? launch_unsplit_as<L, LPC, true, 1>(a, st)
                      : launch_unsplit_as<L, LPC, true, 2>(a, st);
  return phase == 1 ? launch_unsplit_as<L, LPC, false, 1>(a, st)
                    : launch_unsplit_as<L, LPC, false, 2>(a, st);
}

}  // namespace dgb
