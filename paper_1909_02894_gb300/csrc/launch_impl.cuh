// Launch logic of the fused line pass, instantiated once per precision.
#pragma once
#include <cuda_runtime.h>

#include "internal.h"

namespace dgb {

// Elements per thread: FP32 lines of 256 points or more use E = 8 (radix-8 passes; the
// FFT state of a thread fits the 64-register budget of 1024 threads per SM without
// spilling), and so do 64- and 128-point lines in both precisions and FP64 lines of 256..1024
// points (with the fused butterflies 1024^2 0.636 against 0.647 ms per step for E = 16, 512^2
// 0.171 against 0.173, 2048^2 3.01 against 2.82); the other lengths use E = 16.
template <typename T>
constexpr int radix_e(int L) {
  return (sizeof(T) == 4 ? L >= 64 : L >= 64 && L <= 1024) ? 8 : 16;
}
// Elements per thread of the small shape of lines of 128 points or fewer: few, so that a small
// grid's lines spread over many warps. Its pass is bound by the length of each warp's chain
// and, in FP64, by the one warp instruction per 64 cycles that a quarter of an SM takes
// (measured; four warps on different quarters reach the SM's rate of one per 19). Measured per
// step (ms), E = 8 | 4 | 2: complex128 128^2 0.0463 | 0.0276 | 0.0201, 64^2 (0.045) | 0.0237 |
// 0.0165; complex64 128^2 0.0122 | 0.0091 | 0.0085, 64^2 0.0099 | 0.0086 | 0.0074. Many lines
// fill the GPU anyway, and fewer passes win: complex64 128 x 1024 E = 4 0.0136, E = 2 0.0155.
constexpr int radix_small(int L, int n_lines) { return L > 128 ? 0 : n_lines <= 512 ? 2 : 4; }
// The other radix schedule the autotuner may choose (0: none): FP32 lines of 256..4096
// points in radix-16 passes, FP64 lines of 256..1024 points in radix-16, of 2048 points in
// radix-8 passes.
template <typename T>
constexpr int radix_alt(int L) {
  return L < 256 ? 0 : sizeof(T) == 4 ? (L <= 4096 ? 16 : 0) : L <= 1024 ? 16 : L <= 2048 ? 8 : 0;
}

template <typename T, int L, int LPC, int MODE, int E = radix_e<T>(L)>
static cudaError_t launch_one(const LinePassArgs<T>& a, cudaStream_t st) {
  using Gm = Geo<T, L, LPC, E>;
  if (a.n_lines % Gm::GL != 0 || a.n_lines < Gm::GL) return cudaErrorInvalidValue;
  auto kern = line_pass_kernel<T, L, LPC, E, MODE>;
  // Function attributes are per device; set them once per device for this kernel.
  static bool configured[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Gm::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const int grid = (a.inst ? a.inst_capacity : 1) * (a.n_lines / LPC);
  // Programmatic dependent launch saves 0.0023 ms per pass. Not for complex128 passes of
  // several waves, which it made slower (1024^2: 0.755 against 0.734 ms per step; 512^2, one
  // wave: 0.194 against 0.199), nor in a batch's graph, whose kernels start faster without
  // (13 128^2 instances: 0.0179 with, 0.0158 ms per step without).
  const bool pdl = !a.inst && (sizeof(T) == 4 || grid <= 2 * sm_count());
  return launch_pdl(kern, dim3(grid), dim3(Gm::THREADS), Gm::SMEM, st, pdl, Gm::CS, a);
}

// Two CTA shapes per line length (opt 0 smaller, opt 1 larger; 4096-point lines have one).
// Lines per CTA, by precision:
//   FP32 (E = 8 from 256 points): 256: 4|8, 512: 2|4, 1024: 1|2, 2048: 1|2, 4096: 1
//     (256|512 threads, 512|1024 at 2048, 1024 at 4096)
//   FP64 (E = 16 from 2048 points): 256: 1|2, 512: 2|4, 1024: 1|2, 2048: 1|2, 4096: 1 (64..512 threads).
//     The FP64 pass is bound by the FP64 units and its CTAs hold 96-172 registers per
//     thread, so few CTAs fit an SM: small CTAs keep all 152 SMs evenly loaded. Measured (ms per
//     step, opt 0 | opt 1): 256^2 0.0497 | 0.0500, 512^2 0.1717 | 0.1714, 1024^2 0.636 | 0.761,
//     2048^2 3.21 | 2.82.
//   both, 128 points or fewer: as few lines as fill a warp or two with radix_small elements per
//     thread (16 points 4 | 2, 32 points 2 | 1 for E = 4 | 2, 64 and 128 points 1) | 16 lines.
//     A full GPU prefers the larger shape (100 complex64 128^2 instances: 0.074 ms per step
//     against 0.091 with E = 4), which is the batches' default.
template <typename T, int MODE, int E>
static cudaError_t dispatch_small(const LinePassArgs<T>& a, cudaStream_t st) {
  switch (a.L) {
    case 16: return launch_one<T, 16, E, MODE, E>(a, st);
    case 32: return launch_one<T, 32, E / 2, MODE, E>(a, st);
    case 64: return launch_one<T, 64, 1, MODE, E>(a, st);
    case 128: return launch_one<T, 128, 1, MODE, E>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int MODE>
static cudaError_t dispatch(const LinePassArgs<T>& a, int opt, cudaStream_t st) {
  constexpr bool F = sizeof(T) == 4;
  const bool big = (MODE == MODE_STEP) && opt != 0;
  // the derivative mode has no option: the larger shape for many short complex64 lines
  const bool wide = MODE == MODE_STEP ? big
                                      : F && a.L >= 32 && (size_t)a.L * a.n_lines >= kWideShortLines;
  if (!wide && a.L <= 128) {
    if (!a.tw_small) return cudaErrorInvalidValue;
    LinePassArgs<T> b = a;
    b.tw = a.tw_small;
    return radix_small(a.L, a.n_lines) == 2 ? dispatch_small<T, MODE, 2>(b, st)
                                            : dispatch_small<T, MODE, 4>(b, st);
  }
  switch (a.L) {
    case 16: return launch_one<T, 16, 16, MODE>(a, st);
    case 32: return launch_one<T, 32, 16, MODE>(a, st);
    case 64: return launch_one<T, 64, 16, MODE>(a, st);
    case 128: return launch_one<T, 128, 16, MODE>(a, st);
    default: break;
  }
  if (a.L == 4096) return launch_one<T, 4096, 1, MODE>(a, st);
  if constexpr (MODE == MODE_STEP) {
    if (big) {
      switch (a.L) {
        case 256: return launch_one<T, 256, F ? 8 : 2, MODE>(a, st);
        case 512: return launch_one<T, 512, 4, MODE>(a, st);
        case 1024: return launch_one<T, 1024, 2, MODE>(a, st);
        case 2048: return launch_one<T, 2048, 2, MODE>(a, st);
        default: return cudaErrorInvalidValue;
      }
    }
  }
  switch (a.L) {
    case 256: return launch_one<T, 256, F ? 4 : 1, MODE>(a, st);
    case 512: return launch_one<T, 512, 2, MODE>(a, st);
    case 1024: return launch_one<T, 1024, 1, MODE>(a, st);
    case 2048: return launch_one<T, 2048, 1, MODE>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

// The alternative radix schedule (radix_alt), opt 3 the smaller and opt 4 the larger of two
// CTA shapes (about 256 and 512 threads; 1 and 2 lines for FP64 lines of 256 points;
// 4096-point FP32 lines and 2048-point FP64 lines have one, 512 threads). Its twiddle table (a.tw_alt) has the layout of that radix.
template <typename T>
static cudaError_t dispatch_alt(const LinePassArgs<T>& a0, int opt, cudaStream_t st) {
  if (!a0.tw_alt) return cudaErrorInvalidValue;
  LinePassArgs<T> a = a0;
  a.tw = a0.tw_alt;
  const bool big = opt == 4;
  constexpr int M = MODE_STEP;
  if constexpr (sizeof(T) == 4) {  // radix 16: 2 L / 16 threads per line
    switch (a.L) {
      case 256: return big ? launch_one<T, 256, 16, M, 16>(a, st) : launch_one<T, 256, 8, M, 16>(a, st);
      case 512: return big ? launch_one<T, 512, 8, M, 16>(a, st) : launch_one<T, 512, 4, M, 16>(a, st);
      case 1024: return big ? launch_one<T, 1024, 4, M, 16>(a, st) : launch_one<T, 1024, 2, M, 16>(a, st);
      case 2048: return big ? launch_one<T, 2048, 2, M, 16>(a, st) : launch_one<T, 2048, 1, M, 16>(a, st);
      case 4096: return launch_one<T, 4096, 1, M, 16>(a, st);
      default: return cudaErrorInvalidValue;
    }
  } else {  // radix 16 up to 1024 points, radix 8 at 2048
    switch (a.L) {
      case 256: return big ? launch_one<T, 256, 2, M, 16>(a, st) : launch_one<T, 256, 1, M, 16>(a, st);
      case 512: return big ? launch_one<T, 512, 4, M, 16>(a, st) : launch_one<T, 512, 2, M, 16>(a, st);
      case 1024: return big ? launch_one<T, 1024, 2, M, 16>(a, st) : launch_one<T, 1024, 1, M, 16>(a, st);
      case 2048: return launch_one<T, 2048, 1, M, 8>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
}

template <typename T>
cudaError_t launch_line_pass(const LinePassArgs<T>& a, int mode, int opt, cudaStream_t st) {
  if (mode == MODE_DERIV) return dispatch<T, MODE_DERIV>(a, 0, st);
  if (opt == 3 || opt == 4) {
    if (radix_alt<T>(a.L) == 0) return cudaErrorInvalidValue;
    return dispatch_alt<T>(a, opt, st);
  }
  if constexpr (sizeof(T) == 4) {
    if (opt == 2) {
      switch (a.L) {
        case 256: return launch_team<256>(a, st);
        case 512: return launch_team<512>(a, st);
        case 1024: return launch_team<1024>(a, st);
        case 2048: return launch_team<2048>(a, st);
        case 4096: return launch_team<4096>(a, st);
        default: break;
      }
    }
  }
  return dispatch<T, MODE_STEP>(a, opt >= 1 ? 1 : 0, st);
}

template <typename T>
int line_pass_radix(int L) { return radix_e<T>(L); }
template <typename T>
int line_pass_radix_alt(int L) { return radix_alt<T>(L); }
template <typename T>
int line_pass_radix_small(int L, int n_lines) { return radix_small(L, n_lines); }

}  // namespace dgb
