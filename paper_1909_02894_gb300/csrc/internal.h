// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <string>

#include "common.cuh"
#include "line_pass.cuh"

namespace dgb {

// Kernel launch with, if `pdl`, programmatic stream serialization: the kernel may be scheduled
// while its predecessor in the stream still runs (it calls pdl_wait before it touches memory),
// and, if cluster > 1, that cluster size. Loads through the read-only path (__ldg, ld.global.nc)
// need data that no kernel writes while the loading one is resident, which pdl_wait does not
// change: a kernel launched with `pdl` takes that path for tables only (coefficients,
// twiddles, multipliers, instance pointers; their producers are launched without it and are
// complete before), and reads states and terms by ordinary loads or bulk copies.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, bool pdl, int cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

inline int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!cached[dev]) cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev);
  return cached[dev];
}

// Sets the text that dirac_last_error(NULL) returns (errors without a context).
void set_global_error(const std::string& msg);

// Enqueues one fused line pass (MODE_STEP or MODE_DERIV). opt selects the CTA shape:
// 0 = about 256 threads per CTA, 1 = 512 threads, 2 = the radix-16 team pass (complex64
// step mode, lines of 256..4096 points; otherwise as 1).
template <typename T>
cudaError_t launch_line_pass(const LinePassArgs<T>& a, int mode, int opt, cudaStream_t st);
// The team pass runs pairs of lines from this many points per launch (see launch_team_sized).
constexpr size_t kTeamPairPoints = (size_t)1 << 20, kTeamPairPointsBatch = (size_t)1 << 21;
// Elements per thread (8 or 16) the line pass uses for line length L; the twiddle table
// of that axis must be built for the same value.
template <typename T>
int line_pass_radix(int L);
// The alternative radix schedule the autotuner may pick for lines of L points (0: none);
// launch options 3 and 4 run it, with a twiddle table of that radix in tw_alt.
template <typename T>
int line_pass_radix_alt(int L);
// Short complex64 lines (32 to 128 points): from this many points on the larger shape is taken
// (see pass_opt in dirac_api.cu).
constexpr size_t kWideShortLines = (size_t)1 << 17;
// Elements per thread of launch option 0 and of the derivative mode for lines of 128 points
// or fewer (0: longer lines), with a twiddle table of that radix in tw_small.
template <typename T>
int line_pass_radix_small(int L, int n_lines);
// Debug builds (-DDIRAC_DEBUG=1): read and clear the index-check flags of the line-pass
// translation units; nonzero when a check failed. Always 0 in release builds.
int dgb_debug_flag_c64();
int dgb_debug_flag_c128();
int dgb_debug_flag_small();
int dgb_debug_flag_team_256();
int dgb_debug_flag_team_512();
int dgb_debug_flag_team_1024();
int dgb_debug_flag_team_2048();
int dgb_debug_flag_team_4096();
inline int dgb_debug_bounds() {
  return dgb_debug_flag_c64() | dgb_debug_flag_c128() | dgb_debug_flag_team_256() |
         dgb_debug_flag_team_512() | dgb_debug_flag_team_1024() | dgb_debug_flag_team_2048() |
         dgb_debug_flag_team_4096() | dgb_debug_flag_small();
}

// ---- FP64 precompute (precompute.cu)
// a1, a2, meff, w and the two log fields (packed as a complex128 spinor (f1, f2)) from the
// metric; g == nullptr means 1.
cudaError_t launch_metric_fields(const double* g00, const double* g11, const double* g22,
                                 int n, double c, double mass, int conn, double* a1,
                                 double* a2, double* meff, double* w, Q4<double>* logs,
                                 cudaStream_t st);
// Omega_x, Omega_y (normal layout) from the x derivative (transposed layout [nx][ny]) and
// the y derivative (normal layout) of the log fields.
cudaError_t launch_omega(const Q4<double>* dxT, const Q4<double>* dy, int nx, int ny,
                         double fac, double* omx, double* omy, cudaStream_t st);
// 1/S for grid indices of one axis (Sec. 3 profiles), S = 1 + exp(i theta) Sigma~: the real
// part into sinv and, if sinv_im is not null, the imaginary part (else theta must be 0).
cudaError_t launch_pml(int n, double a, int width, int type, double sigma0, double theta,
                       double* sinv, double* sinv_im, cudaStream_t st);
// beta1 = a1/S1 - 1 (normal layout), beta2T = a2/S2 - 1 (transposed layout), in T; with
// complex stretching (sxinv_im, syinv_im not null) the imaginary parts go to beta1_im,
// beta2T_im.
template <typename T>
cudaError_t launch_beta(const double* a1, const double* a2, const double* sxinv,
                        const double* syinv, const double* sxinv_im, const double* syinv_im,
                        int nx, int ny, T* beta1, T* beta2T, T* beta1_im, T* beta2T_im,
                        cudaStream_t st);
// Half-step matrices for dt: U (normal layout), U and U^2 (transposed layout) and, if
// u2_n is not null, U^2 in the normal layout, stored as (c0 - 1, c1, c2, c3) in T.
template <typename T>
cudaError_t launch_halfstep(const double* a1, const double* a2, const double* meff,
                            const double* omx, const double* omy, int nx, int ny, double dt,
                            Q4<T>* u_n, Q4<T>* u_t, Q4<T>* u2_t, Q4<T>* u2_n,
                            cudaStream_t st);
// Per-axis tables: per-pass twiddle blocks (layout in line_pass.cuh); step multipliers
// ((cos(dt xi) - 1)/n, sin(dt xi)/n) as hi/lo pairs; derivative multipliers xi/n.
template <typename T>
cudaError_t launch_twiddles(int n, int e, Cx<T>* tw, cudaStream_t st);
template <typename T>
cudaError_t launch_step_mult(int n, double a, double dt, Q4<T>* mult, cudaStream_t st);
// Team pass (lines of n = 256..4096 points): a multiplier table in its order, its twiddles.
template <typename T>
cudaError_t launch_team_perm(int n, const Q4<T>* src, Q4<T>* dst, cudaStream_t st);
template <typename T>
cudaError_t launch_team_twiddles(int n, Cx<T>* tw, cudaStream_t st);
template <typename T>
cudaError_t launch_deriv_mult(int n, double a, Q4<T>* mult, cudaStream_t st);

// Half step with static potentials: general complex U and U^2 per point (two Q4 per point
// holding U - I: (d00, u01), (u10, d11)), in the normal or the transposed layout; V, Ax, Ay may
// be null (0).
template <typename T>
cudaError_t launch_halfstep_general(const double* a1, const double* a2, const double* meff,
                                    const double* omx, const double* omy, const double* V,
                                    const double* Ax, const double* Ay, int nx, int ny,
                                    double dt, bool transposed, Q4<T>* ug, Q4<T>* ug2,
                                    cudaStream_t st);
// psi <- U psi (psi in the normal layout) for such a general U in the normal and in the
// transposed layout.
template <typename T>
cudaError_t launch_apply_ug(Q4<T>* psi, const Q4<T>* ug, size_t n, cudaStream_t st);
template <typename T>
cudaError_t launch_apply_ug_t(Q4<T>* psi, const Q4<T>* ug_t, int nx, int ny, cudaStream_t st);

// The team pass for one line length (256..4096; one translation unit each, team_<L>.cu), and
// one phase (1 or 2) of the unsplit operator.
template <int L>
cudaError_t launch_team(const LinePassArgs<float>& a, cudaStream_t st);
template <int L>
cudaError_t launch_team_unsplit(const UnsplitArgs& a, int phase, cudaStream_t st);
// One phase of the unsplit operator on complex64 rows of L = 256..4096 points.
cudaError_t launch_unsplit(const UnsplitArgs& a, int L, int phase, cudaStream_t st);

// ---- small grids (small_steps.cu): n Scheme II steps of a complex64 grid in one launch, where
// both axes have 64 or 128 points (small_steps_grid). lead / trail: U before the first / after
// the last step (U^2 otherwise and between). cudaErrorNotSupported if no cluster of the needed
// size fits the device.
struct SmallStepArgs {
  Q4<float>* psi;       // [ny][nx], updated in place
  const float* beta1;   // b^1 - 1 [ny][nx]
  const float* beta2;   // b^2 - 1 [nx][ny]
  const Q4<float>* u_n;   // U [ny][nx], U and U^2 [nx][ny]; all null when U = I
  const Q4<float>* u_t;
  const Q4<float>* u2_t;
  const Q4<float>* mult_x;
  const Q4<float>* mult_y;
  const Cx<float>* tw_x;  // launch_twiddles with 8 elements per thread
  const Cx<float>* tw_y;
};
bool small_steps_grid(int nx, int ny);
cudaError_t launch_small_steps(const SmallStepArgs& a, int nx, int ny, int n, bool lead,
                               bool trail, cudaStream_t st);

// ---- unsplit polynomial scheme (unsplit.cu)
// psi <- U psi at every point (normal layout).
template <typename T>
cudaError_t launch_apply_u(Q4<T>* psi, const Q4<T>* u, size_t n, cudaStream_t st);
// out = alpha (b1 sigma_x dx + b2 sigma_y dy) + gamma base + beta prev (base and prev may
// be null); b^j = a^j / S^j from the FP64 fields (complex when the
// imaginary parts of 1/S are given); all normal layout.
template <typename T>
cudaError_t launch_unsplit_combine(const Q4<T>* dx, const Q4<T>* dy, const double* a1,
                                   const double* a2, const double* sxinv, const double* syinv,
                                   const double* sxinv_im, const double* syinv_im, int nx,
                                   int ny, double ar, double ai, const Q4<T>* base, double gr,
                                   double gi, const Q4<T>* prev, double beta, Q4<T>* out,
                                   cudaStream_t st);
// Per-block maxima of |b1|, |b2| into partials[2 * n_blocks].
cudaError_t launch_max_b(const double* a1, const double* a2, const double* sxinv,
                         const double* syinv, const double* sxinv_im, const double* syinv_im,
                         int nx, int ny, double* partials, int n_blocks, cudaStream_t st);
// Krylov building blocks (Scheme I); V is a device array of count vector pointers, every
// launch uses at most n_blocks blocks per chunk of vectors and leaves its sums, added in a fixed
// order, in device memory (partials: 2 n_blocks count doubles; ticket: a zeroed counter).
// kind 0: dots[2 i] = <V_i, w> (re, im);
// kind 1: w -= sum_i coef_i V_i, then dots as for kind 0 (count <= 4);
// kind 2: w -= sum_i coef_i V_i, then dots[0] = <w, w>, dots[1] = 1 / sqrt(dots[0]) (1 unless
// dots[0] > 0).
// fp64: complex64 vectors summed in FP64 too (slower, for squares beyond the FP32 range).
template <typename T>
cudaError_t launch_gram_schmidt(int kind, bool fp64, const Q4<T>* const* V, int count, Q4<T>* w,
                                const double* coef, size_t n, double* partials, unsigned* ticket,
                                double* dots, int n_blocks, cudaStream_t st);
// v = 2 (rhs - x) (mode 0) or rhs - v (mode 1); dots[0] = <v, v>, dots[1] = <rhs, rhs> (mode 0),
// dots[2] = 1 / sqrt(dots[0]) (1 unless dots[0] > 0).
template <typename T>
cudaError_t launch_residual(int mode, const Q4<T>* rhs, const Q4<T>* x, Q4<T>* v, size_t n,
                            double* partials, unsigned* ticket, double* dots, int n_blocks,
                            cudaStream_t st);
// v *= dots[at] (device memory); dots[0..at) and the device error flag *err also go to host and
// *host_err (pinned host memory).
template <typename T>
cudaError_t launch_normalise(Q4<T>* v, const double* dots, int at, const int* err, double* host,
                             double* host_err, size_t n, cudaStream_t st);
// out += sum_i coef_i V_i with complex FP64 coef (device array of 2 count doubles).
template <typename T>
cudaError_t launch_multi_axpy(Q4<T>* out, const Q4<T>* const* V, const double* coef, int count,
                              size_t n, cudaStream_t st);
// J_0(x) .. J_n(x) into out[0..n] (host, FP64); false for x < 0 or n < 0.
bool bessel_j_series(double x, int n, double* out);

// Tiled transpose of a [rows][cols] array of Q4<T> into [cols][rows].
template <typename T>
cudaError_t launch_transpose(const Q4<T>* in, Q4<T>* out, int rows, int cols, cudaStream_t st);

// ---- state conversion and observables (observables.cu)
// psi[k] = (p1[k], p2[k]) from a [2][n] complex128 array, and back.
template <typename T>
cudaError_t launch_pack(const double* src, Q4<T>* psi, size_t n, cudaStream_t st);
template <typename T>
cudaError_t launch_unpack(const Q4<T>* psi, double* dst, size_t n, cudaStream_t st);
// Per-block FP64 partial sums {norm, norm_gamma, e_re, e_im} into partials[blocks][4]
// and the density map (if not null). dx and dy may be null (no energy); the static
// potentials V, Ax, Ay may be null (0).
template <typename T>
cudaError_t launch_observables(const Q4<T>* psi, const Q4<T>* dx, const Q4<T>* dy,
                               const double* a1, const double* a2, const double* meff,
                               const double* w, const double* omx, const double* omy,
                               const double* V, const double* Ax, const double* Ay,
                               size_t n, double* density, double* partials, int blocks,
                               cudaStream_t st);
cudaError_t launch_reduce_partials(const double* partials, int blocks, double scale,
                                   double* result, cudaStream_t st);
int observables_blocks(size_t n);

}  // namespace dgb
