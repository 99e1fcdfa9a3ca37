// The unsplit operator on complex64 states (team_unsplit.cuh): launch rule.
#include <cuda_runtime.h>

#include "internal.h"
#include "team_unsplit.cuh"

namespace dgb {

static int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev]) cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev);
  return cached[dev];
}

template <int L, int LPC, bool PAIR, int PHASE>
static cudaError_t launch_as(const UnsplitArgs& a, cudaStream_t st) {
  using G = TGeo<L, LPC, PAIR>;
  if (!a.in || !a.out || !a.beta || !a.tw || !a.mult || !a.err || a.n_lines % G::LPU != 0 ||
      (PHASE == 1 && !a.out_in) || (PHASE == 2 && !a.s_other))
    return cudaErrorInvalidValue;
  auto kern = line_pass_team_unsplit<L, LPC, PAIR, PHASE>;
  static bool configured[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const int units = a.n_lines / G::LPU;
  const int ctas = (units + G::GROUPS - 1) / G::GROUPS, most = G::MINB * sm_count();
  return launch_pdl(kern, dim3(ctas < most ? ctas : most), dim3(G::THREADS), G::SMEM, st, true, 0,
                    a, units);
}

// Pairs of lines from 2^20 points, as for the step pass (launch_team_sized).
template <int L>
static cudaError_t launch_sized(const UnsplitArgs& a, int phase, cudaStream_t st) {
  constexpr int LPC = L >= 2048 ? 1 : 2048 / L;
  if ((size_t)a.n_lines * L >= kTeamPairPoints)
    return phase == 1 ? launch_as<L, LPC, true, 1>(a, st) : launch_as<L, LPC, true, 2>(a, st);
  return phase == 1 ? launch_as<L, LPC, false, 1>(a, st) : launch_as<L, LPC, false, 2>(a, st);
}

cudaError_t launch_unsplit(const UnsplitArgs& a, int L, int phase, cudaStream_t st) {
  if (phase != 1 && phase != 2) return cudaErrorInvalidValue;
  switch (L) {
    case 256: return launch_sized<256>(a, phase, st);
    case 512: return launch_sized<512>(a, phase, st);
    case 1024: return launch_sized<1024>(a, phase, st);
    case 2048: return launch_sized<2048>(a, phase, st);
    case 4096: return launch_sized<4096>(a, phase, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dgb
