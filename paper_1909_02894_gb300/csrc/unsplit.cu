// Pointwise kernels of the unsplit polynomial scheme (Sec. 4.2 eq. op_split_poly, Sec. 5
// eq. poly): the middle step applies sum_q a_q P_q(dt A) with
//   A psi = - sum_j b^j sigma_j [[d_j]] psi,   b^j = a^j / S^j (Sec. 3),
// where the spectral derivatives come from the derivative-mode line passes and the rest
// is one combine kernel per operator application.
#include <cuda_runtime.h>
#include <math.h>

#include "internal.h"

namespace dgb {

namespace {
constexpr int TPB = 256;
unsigned blocks_for(size_t n) { return (unsigned)((n + TPB - 1) / TPB); }
}  // namespace

// psi <- U psi at every point of the normal layout
template <typename T>
__global__ void k_apply_u(Q4<T>* psi, const Q4<T>* u, size_t n) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) psi[k] = apply_u(u[k], psi[k]);
}

// psi <- U psi for a general complex U stored as two Q4 per point (deviation from I):
// (d00, u01), (u10, d11)
template <typename T>
__global__ void k_apply_ug(Q4<T>* psi, const Q4<T>* ug, size_t n) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  psi[k] = apply_u_general(ug[2 * k], ug[2 * k + 1], psi[k]);
}

// S = b1 sigma_x dx + b2 sigma_y dy with sigma_x (u, v) = (v, u), sigma_y (u, v) =
// (-i v, i u); out = alpha S + gamma base + beta prev.
// b^j complex with complex stretching (sxinv_im, syinv_im not null).
template <typename T>
__global__ void k_unsplit_combine(const Q4<T>* dx, const Q4<T>* dy, const double* a1,
                                  const double* a2, const double* sxinv, const double* syinv,
                                  const double* sxinv_im, const double* syinv_im, int nx,
                                  int ny, T ar, T ai, const Q4<T>* base, T gr, T gi,
                                  const Q4<T>* prev, T beta, Q4<T>* out) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (size_t)nx * ny) return;
  const int j = (int)(k / nx), i = (int)(k - (size_t)j * nx);
  const T b1 = (T)(a1[k] * sxinv[i]), b2 = (T)(a2[k] * syinv[j]);
  const T b1i = sxinv_im ? (T)(a1[k] * sxinv_im[i]) : T(0);
  const T b2i = syinv_im ? (T)(a2[k] * syinv_im[j]) : T(0);
  const Q4<T> x = dx[k], y = dy[k];
  // sigma_x dx = (dx2, dx1), sigma_y dy = (-i dy2, i dy1), times complex b
  const T t1r = y.w, t1i = -y.z, t2r = -y.y, t2i = y.x;  // sigma_y dy components
  const T s1r = (b1 * x.z - b1i * x.w) + (b2 * t1r - b2i * t1i);
  const T s1i = (b1 * x.w + b1i * x.z) + (b2 * t1i + b2i * t1r);
  const T s2r = (b1 * x.x - b1i * x.y) + (b2 * t2r - b2i * t2i);
  const T s2i = (b1 * x.y + b1i * x.x) + (b2 * t2i + b2i * t2r);
  Q4<T> o = {ar * s1r - ai * s1i, ar * s1i + ai * s1r, ar * s2r - ai * s2i, ar * s2i + ai * s2r};
  if (base) {
    const Q4<T> p = base[k];
    o.x += gr * p.x - gi * p.y;
    o.y += gr * p.y + gi * p.x;
    o.z += gr * p.z - gi * p.w;
    o.w += gr * p.w + gi * p.z;
  }
  if (prev) {
    const Q4<T> p = prev[k];
    o.x += beta * p.x;
    o.y += beta * p.y;
    o.z += beta * p.z;
    o.w += beta * p.w;
  }
  out[k] = o;
}

// Per-block maxima of |b1| and |b2| (grid-stride), partials[2 b], partials[2 b + 1].
__global__ void k_max_b(const double* a1, const double* a2, const double* sxinv,
                        const double* syinv, const double* sxinv_im, const double* syinv_im,
                        int nx, int ny, double* partials) {
  __shared__ double m1[TPB], m2[TPB];
  double x1 = 0.0, x2 = 0.0;
  const size_t n = (size_t)nx * ny;
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(k / nx), i = (int)(k - (size_t)j * nx);
    x1 = fmax(x1, fabs(a1[k]) * hypot(sxinv[i], sxinv_im ? sxinv_im[i] : 0.0));
    x2 = fmax(x2, fabs(a2[k]) * hypot(syinv[j], syinv_im ? syinv_im[j] : 0.0));
  }
  m1[threadIdx.x] = x1;
  m2[threadIdx.x] = x2;
  __syncthreads();
  for (int s = TPB / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      m1[threadIdx.x] = fmax(m1[threadIdx.x], m1[threadIdx.x + s]);
      m2[threadIdx.x] = fmax(m2[threadIdx.x], m2[threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = m1[0];
    partials[2 * blockIdx.x + 1] = m2[0];
  }
}

// ---- Krylov building blocks (Scheme I): complex inner products <V_i, w> = sum conj(V_i) w
// over both components, accumulated beyond the state's precision.
//
// FP64 states: FP64 fused multiply-adds. FP32 states: the FP64 pipe (two lanes per SM and
// clock, conversions included) made a product of two vectors cost 14 us at 512^2, four times
// its memory traffic; instead each product is split exactly into its FP32 rounding and the
// remainder (an FMA), and both are added to a sum of three FP32 terms by two-sums (Knuth; the
// scheme of Ogita, Rump and Oishi's DotK with K = 3, threefold FP32 precision), within 8
// points of a thread and across the 32 lanes of a warp; everything beyond is added in FP64.
// Error of a product of unit vectors against the exact sum, 4096 to 2^18 points (noise and wave
// packets, emulated in tests/test_krylov_sums_cpu.py): at most one FP64 rounding, 1.1e-16.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<double> {
  double d = 0.0;
  __device__ __forceinline__ void add(double a, double b) { d += a * b; }
  __device__ __forceinline__ void sub(double a, double b) { d -= a * b; }
  __device__ __forceinline__ void flush() {}
  // the warp's sum (valid in lane 0); `flushed` (uniform): flush has been called
  __device__ __forceinline__ double warp_total(bool) {
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    return d;
  }
};
template <>
struct DotAcc<float> {
  double d = 0.0;
  float s = 0.f, c = 0.f, g = 0.f;
  // x <- the rounded x + p; returns the rounding error exactly
  static __device__ __forceinline__ float two_sum(float& x, float p) {
    const float t = __fadd_rn(x, p), z = __fsub_rn(t, x);
    const float r = __fadd_rn(__fsub_rn(x, __fsub_rn(t, z)), __fsub_rn(p, z));
    x = t;
    return r;
  }
  // the sum of hi + lo, lo at the scale of hi's rounding
  __device__ __forceinline__ void add_pair(float hi, float lo) {
    const float r1 = two_sum(s, hi), r2 = two_sum(lo, r1), r3 = two_sum(c, lo);
    g = __fadd_rn(g, __fadd_rn(r2, r3));
  }
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    add_pair(p, __fmaf_rn(a, b, -p));
  }
  __device__ __forceinline__ void sub(float a, float b) { add(-a, b); }
  __device__ __forceinline__ void flush() {
    d += (double)s + ((double)c + (double)g);
    s = c = g = 0.f;
  }
  __device__ __forceinline__ double warp_total(bool flushed) {
    for (int o = 16; o > 0; o >>= 1) {
      const float ps = __shfl_down_sync(0xffffffffu, s, o);
      const float pc = __shfl_down_sync(0xffffffffu, c, o);
      const float pg = __shfl_down_sync(0xffffffffu, g, o);
      add_pair(ps, pc);
      g = __fadd_rn(g, pg);
    }
    if (flushed)
      for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    return (threadIdx.x & 31) == 0 ? d + ((double)s + ((double)c + (double)g)) : 0.0;
  }
};
template <typename A, typename T>
__device__ __forceinline__ void dot_point(DotAcc<A>& re, DotAcc<A>& im, const Q4<T>& a,
                                          const Q4<T>& b) {
  re.add(a.x, b.x);
  re.add(a.y, b.y);
  re.add(a.z, b.z);
  re.add(a.w, b.w);
  im.add(a.x, b.y);
  im.sub(a.y, b.x);
  im.add(a.z, b.w);
  im.sub(a.w, b.z);
}
template <typename A, typename T>
__device__ __forceinline__ void norm_point(DotAcc<A>& re, const Q4<T>& a) {
  re.add(a.x, a.x);
  re.add(a.y, a.y);
  re.add(a.z, a.z);
  re.add(a.w, a.w);
}

// Sums `count` values per block (accumulators acc[i] of each thread) into partials[i gridDim.x +
// block]; the grid's last block to finish adds the blocks' partial sums, in the order of a
// fixed tree, into result[i], and resets the ticket. total: values over all gridDim.y chunks;
// first: this chunk's first value. INV: result[total] = 1 / sqrt(result[0]), or 1 unless
// result[0] > 0.
template <int N, bool INV, typename A>
__device__ __forceinline__ void grid_sums(DotAcc<A> (&acc)[N], bool flushed, int count, int first,
                                          int total, double* partials, unsigned* ticket,
                                          double* result) {
  __shared__ double sh[N][TPB / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < count) {
      const double v = acc[i].warp_total(flushed);
      if (lane == 0) sh[i][wid] = v;
    }
  __syncthreads();
  if ((int)threadIdx.x < count) {
    double v = 0.0;
    for (int t = 0; t < TPB / 32; ++t) v += sh[threadIdx.x][t];
    partials[(size_t)(first + threadIdx.x) * gridDim.x + blockIdx.x] = v;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = wid; i < total; i += TPB / 32) {
    double v = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(partials + (size_t)i * gridDim.x + b);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) result[i] = v;
  }
  if constexpr (INV) {
    __syncthreads();
    if (threadIdx.x == 0) result[total] = result[0] > 0.0 ? 1.0 / sqrt(result[0]) : 1.0;
  }
  if (threadIdx.x == 0) *ticket = 0;
}

constexpr int kChunk = 4;  // vectors whose products a thread accumulates at once

// KIND 0: dots of the chunk's vectors with w. KIND 1 (one chunk): w -= sum coef_i V_i first.
// KIND 2 (grid.y = 1): w -= sum coef_i V_i over all `count` vectors, then the norm of w.
// Products and norms in accumulators of type A: T's own, or FP64 for complex64 vectors whose
// squares left the FP32 range.
template <typename T, typename A, int KIND>
__global__ void __launch_bounds__(TPB) k_gram_schmidt(const Q4<T>* const* V, int count, Q4<T>* w,
                                                      const double* coef, size_t n,
                                                      double* partials, unsigned* ticket,
                                                      double* dots) {
  const int first = KIND == 0 ? blockIdx.y * kChunk : 0;
  const int c = KIND == 2 ? count : min(kChunk, count - first);
  DotAcc<A> acc[KIND == 2 ? 1 : 2 * kChunk];  // re, im of each product; the norm
  int since = 0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const bool flushed = n > 8 * stride;
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
    Q4<T> x = w[k];
    if constexpr (KIND == 2) {
      for (int i = 0; i < c; ++i) {
        const T cr = (T)-coef[2 * i], ci = (T)-coef[2 * i + 1];
        const Q4<T> v = V[i][k];
        x.x += cr * v.x - ci * v.y;
        x.y += cr * v.y + ci * v.x;
        x.z += cr * v.z - ci * v.w;
        x.w += cr * v.w + ci * v.z;
      }
      w[k] = x;
      norm_point(acc[0], x);
    } else {
      Q4<T> v[kChunk];
#pragma unroll
      for (int i = 0; i < kChunk; ++i)
        if (i < c) v[i] = V[first + i][k];
      if constexpr (KIND == 1) {
#pragma unroll
        for (int i = 0; i < kChunk; ++i)
          if (i < c) {
            const T cr = (T)-coef[2 * i], ci = (T)-coef[2 * i + 1];
            x.x += cr * v[i].x - ci * v[i].y;
            x.y += cr * v[i].y + ci * v[i].x;
            x.z += cr * v[i].z - ci * v[i].w;
            x.w += cr * v[i].w + ci * v[i].z;
          }
        w[k] = x;
      }
#pragma unroll
      for (int i = 0; i < kChunk; ++i)
        if (i < c) dot_point(acc[2 * i], acc[2 * i + 1], v[i], x);
    }
    if (flushed && ++since == 8) {
      since = 0;
#pragma unroll
      for (int i = 0; i < (KIND == 2 ? 1 : 2 * kChunk); ++i) acc[i].flush();
    }
  }
  if constexpr (KIND == 2)
    grid_sums<1, true>(acc, flushed, 1, 0, 1, partials, ticket, dots);
  else
    grid_sums<2 * kChunk, false>(acc, flushed, 2 * c, 2 * first, 2 * count, partials, ticket, dots);
}

// FP64 sums in both precisions: these vectors carry the state's own scale, whose squares may
// leave the FP32 range (the basis vectors above have unit norm).
template <typename T>
__global__ void __launch_bounds__(TPB) k_residual(int mode, const Q4<T>* rhs, const Q4<T>* x,
                                                  Q4<T>* v, size_t n, double* partials,
                                                  unsigned* ticket, double* dots) {
  DotAcc<double> acc[2];
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
    const Q4<T> b = rhs[k], q = mode == 0 ? x[k] : v[k];
    const T f = mode == 0 ? T(2) : T(1);
    const Q4<T> r = {f * (b.x - q.x), f * (b.y - q.y), f * (b.z - q.z), f * (b.w - q.w)};
    v[k] = r;
    norm_point(acc[0], r);
    if (mode == 0) norm_point(acc[1], b);
  }
  grid_sums<2, true>(acc, true, 2, 0, 2, partials, ticket, dots);
}

// v *= dots[at]; dots[0..at) and the device error flag go to pinned host memory, written from
// here as a copy of its own behind this kernel delayed the host, which waits for these values
// (Scheme I at 512^2, 4 steps with set_state and get_state: 1.43 -> 1.31 ms).
template <typename T>
__global__ void k_normalise(Q4<T>* v, const double* dots, int at, const int* err, double* host,
                            double* host_err, size_t n) {
  if (blockIdx.x == 0) {
    for (int t = threadIdx.x; t < at; t += TPB) host[t] = dots[t];
    if (threadIdx.x == 0) *host_err = *err;
  }
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const T c = (T)dots[at];
  const Q4<T> p = v[k];
  v[k] = {c * p.x, c * p.y, c * p.z, c * p.w};
}

// out += sum_i c_i V_i (c complex, coef[2 i], coef[2 i + 1]; FP64 coefficients)
template <typename T>
__global__ void k_multi_axpy(Q4<T>* out, const Q4<T>* const* V, const double* coef, int count,
                             size_t n) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  Q4<T> o = out[k];
  for (int i = 0; i < count; ++i) {
    const T cr = (T)coef[2 * i], ci = (T)coef[2 * i + 1];
    const Q4<T> v = V[i][k];
    o.x += cr * v.x - ci * v.y;
    o.y += cr * v.y + ci * v.x;
    o.z += cr * v.z - ci * v.w;
    o.w += cr * v.w + ci * v.z;
  }
  out[k] = o;
}

// Blocks of a reduction over n points: four points per thread (the sums across threads cost as
// much as several points), at most n_max.
static int sum_blocks(size_t n, int n_max) {
  const size_t b = (n + 4 * TPB - 1) / (4 * TPB);
  return (int)(b < (size_t)n_max ? b : (size_t)n_max);
}

template <typename T, typename A>
static void gram_schmidt_as(int kind, const Q4<T>* const* V, int count, Q4<T>* w,
                            const double* coef, size_t n, double* partials, unsigned* ticket,
                            double* dots, int n_blocks, cudaStream_t st) {
  if (kind == 0)
    k_gram_schmidt<T, A, 0><<<dim3(n_blocks, (count + kChunk - 1) / kChunk), TPB, 0, st>>>(
        V, count, w, coef, n, partials, ticket, dots);
  else if (kind == 1)
    k_gram_schmidt<T, A, 1><<<n_blocks, TPB, 0, st>>>(V, count, w, coef, n, partials, ticket, dots);
  else
    k_gram_schmidt<T, A, 2><<<n_blocks, TPB, 0, st>>>(V, count, w, coef, n, partials, ticket, dots);
}

template <typename T>
cudaError_t launch_gram_schmidt(int kind, bool fp64, const Q4<T>* const* V, int count, Q4<T>* w,
                                const double* coef, size_t n, double* partials, unsigned* ticket,
                                double* dots, int n_blocks, cudaStream_t st) {
  if (count < 1 || (kind == 1 && count > kChunk)) return cudaErrorInvalidValue;
  n_blocks = sum_blocks(n, n_blocks);
  if (fp64)
    gram_schmidt_as<T, double>(kind, V, count, w, coef, n, partials, ticket, dots, n_blocks, st);
  else
    gram_schmidt_as<T, T>(kind, V, count, w, coef, n, partials, ticket, dots, n_blocks, st);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_residual(int mode, const Q4<T>* rhs, const Q4<T>* x, Q4<T>* v, size_t n,
                            double* partials, unsigned* ticket, double* dots, int n_blocks,
                            cudaStream_t st) {
  n_blocks = sum_blocks(n, n_blocks);
  k_residual<T><<<n_blocks, TPB, 0, st>>>(mode, rhs, x, v, n, partials, ticket, dots);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_normalise(Q4<T>* v, const double* dots, int at, const int* err, double* host,
                             double* host_err, size_t n, cudaStream_t st) {
  k_normalise<T><<<blocks_for(n), TPB, 0, st>>>(v, dots, at, err, host, host_err, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_multi_axpy(Q4<T>* out, const Q4<T>* const* V, const double* coef, int count,
                              size_t n, cudaStream_t st) {
  k_multi_axpy<T><<<blocks_for(n), TPB, 0, st>>>(out, V, coef, count, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_apply_ug(Q4<T>* psi, const Q4<T>* ug, size_t n, cudaStream_t st) {
  k_apply_ug<T><<<blocks_for(n), TPB, 0, st>>>(psi, ug, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_apply_u(Q4<T>* psi, const Q4<T>* u, size_t n, cudaStream_t st) {
  k_apply_u<T><<<blocks_for(n), TPB, 0, st>>>(psi, u, n);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_unsplit_combine(const Q4<T>* dx, const Q4<T>* dy, const double* a1,
                                   const double* a2, const double* sxinv, const double* syinv,
                                   const double* sxinv_im, const double* syinv_im, int nx,
                                   int ny, double ar, double ai, const Q4<T>* base, double gr,
                                   double gi, const Q4<T>* prev, double beta, Q4<T>* out,
                                   cudaStream_t st) {
  k_unsplit_combine<T><<<blocks_for((size_t)nx * ny), TPB, 0, st>>>(
      dx, dy, a1, a2, sxinv, syinv, sxinv_im, syinv_im, nx, ny, (T)ar, (T)ai, base, (T)gr, (T)gi,
      prev, (T)beta, out);
  return cudaGetLastError();
}

cudaError_t launch_max_b(const double* a1, const double* a2, const double* sxinv,
                         const double* syinv, const double* sxinv_im, const double* syinv_im,
                         int nx, int ny, double* partials, int n_blocks, cudaStream_t st) {
  k_max_b<<<n_blocks, TPB, 0, st>>>(a1, a2, sxinv, syinv, sxinv_im, syinv_im, nx, ny, partials);
  return cudaGetLastError();
}

cudaError_t launch_unsplit(const UnsplitArgs& a, int L, int phase, cudaStream_t st) {
  if (phase != 1 && phase != 2) return cudaErrorInvalidValue;
  switch (L) {
    case 256: return launch_team_unsplit<256>(a, phase, st);
    case 512: return launch_team_unsplit<512>(a, phase, st);
    case 1024: return launch_team_unsplit<1024>(a, phase, st);
    case 2048: return launch_team_unsplit<2048>(a, phase, st);
    case 4096: return launch_team_unsplit<4096>(a, phase, st);
    default: return cudaErrorInvalidValue;
  }
}

// Bessel functions J_0(x) .. J_n(x), x >= 0, by downward recurrence from an order well
// above max(n, x) (where the minimal solution dominates), J_{k-1} = (2k/x) J_k - J_{k+1},
// normalised by the Neumann sum J_0 + 2 (J_2 + J_4 + ...) = 1. Returns false for bad input.
bool bessel_j_series(double x, int n, double* out) {
  if (!(x >= 0.0) || n < 0) return false;
  for (int k = 0; k <= n; ++k) out[k] = 0.0;
  if (x == 0.0) {
    out[0] = 1.0;
    return true;
  }
  const double big = fmax((double)n, x);
  int top = (int)(big + 50.0 + 6.0 * sqrt(big));
  if (top % 2) ++top;
  double hi = 0.0, mid = 1e-300, norm = 0.0;
  for (int k = top; k > 0; --k) {
    const double lo = 2.0 * k / x * mid - hi;  // J_{k-1} (unnormalised)
    hi = mid;
    mid = lo;
    const int idx = k - 1;
    if (fabs(mid) > 1e200) {
      hi *= 1e-200;
      mid *= 1e-200;
      norm *= 1e-200;
      for (int t = 0; t <= n; ++t) out[t] *= 1e-200;
    }
    if (idx <= n) out[idx] = mid;
    if (idx > 0 && idx % 2 == 0) norm += 2.0 * mid;
  }
  norm += mid;
  for (int k = 0; k <= n; ++k) out[k] /= norm;
  return true;
}

#define INST(T)                                                                              \
  template cudaError_t launch_apply_u<T>(Q4<T>*, const Q4<T>*, size_t, cudaStream_t);        \
  template cudaError_t launch_apply_ug<T>(Q4<T>*, const Q4<T>*, size_t, cudaStream_t);       \
  template cudaError_t launch_unsplit_combine<T>(                                            \
      const Q4<T>*, const Q4<T>*, const double*, const double*, const double*, const double*, \
      const double*, const double*, int, int, double, double, const Q4<T>*, double, double,  \
      const Q4<T>*, double, Q4<T>*, cudaStream_t);                                           \
  template cudaError_t launch_gram_schmidt<T>(int, bool, const Q4<T>* const*, int, Q4<T>*,    \
                                              const double*, size_t, double*, unsigned*,      \
                                              double*, int, cudaStream_t);                    \
  template cudaError_t launch_residual<T>(int, const Q4<T>*, const Q4<T>*, Q4<T>*, size_t,    \
                                          double*, unsigned*, double*, int, cudaStream_t);    \
  template cudaError_t launch_normalise<T>(Q4<T>*, const double*, int, const int*, double*,   \
                                           double*, size_t, cudaStream_t);                    \
  template cudaError_t launch_multi_axpy<T>(Q4<T>*, const Q4<T>* const*, const double*, int,  \
                                            size_t, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace dgb
