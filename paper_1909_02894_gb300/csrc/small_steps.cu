// Whole steps of small complex64 grids (axes of 64 or 128 points) inside one launch.
//
// A pass over such a grid takes less time than launching it: 128^2 in two launches per step,
// overlapped by programmatic dependent launch, costs 8.4 us per step, of which the passes'
// arithmetic is well below 1 us. Here one cluster of NC CTAs keeps the grid in shared memory
// for all steps of a call: CTA r holds LY/NC rows for the x passes and LX/NC columns for the y
// passes, a pass writes its finished points straight into the shared memory of the CTA that
// owns them in the other layout (distributed shared memory), and the hardware cluster barrier
// separates the passes. Two state buffers, so one barrier per pass is enough: a pass reads the
// one and writes the other, which nobody reads until the barrier. Each line is transformed
// by L/4 threads of one warp (8 points of one eigencomponent per thread, radix-8 Stockham
// passes, no CTA barrier); b - 1, U^2 and the tables stay in shared memory.
// The arithmetic is that of line_pass_kernel with E = 8, so the results equal, bit for bit,
// those of the batches' default shape. Bound by the latency of each line's chain, the remote
// stores and the cluster barrier. Measured per step: 64^2 0.0074 -> 0.0027 ms, 128 x 64 0.0034,
// 128^2 0.0084 -> 0.0053 (against two launches with 2 points per thread).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace dgb {

namespace {

template <int L>
using SGeo = Geo<float, L, 32 / (L / 4) < 4 ? 4 : 32 / (L / 4), 8>;  // only its line layout is used

template <int LX, int LY, int NC>
struct SPlan {
  static constexpr int ROWS = LY / NC, COLS = LX / NC;  // lines of this CTA in x and y passes
  static constexpr int THREADS = ROWS * (LX / 4);
  static constexpr int PX = LX + 1, PY = LY + 1;  // line pitch (points) of the state buffers
  static constexpr size_t A = 0, B = A + (size_t)ROWS * PX * 16;
  static constexpr size_t U2 = B + (size_t)COLS * PY * 16;
  static constexpr size_t MX = U2 + (size_t)COLS * LY * 16, MY = MX + (size_t)LX * 16;
  static constexpr size_t B1 = MY + (size_t)LY * 16, B2 = B1 + (size_t)ROWS * LX * 4;
  static constexpr size_t FFT = B2 + (size_t)COLS * LY * 4;
  static constexpr size_t FX = (size_t)ROWS * SGeo<LX>::STRIDE * 8;
  static constexpr size_t FY = (size_t)COLS * SGeo<LY>::STRIDE * 8;
  static constexpr size_t SMEM = FFT + (FX > FY ? FX : FY);
  static_assert(ROWS * LX == COLS * LY && THREADS % 32 == 0, "the same threads in both passes");
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

// fft_passes of line_pass.cuh for a line inside one warp
template <int L, bool INV, int P = 0, int NS = 1>
__device__ __forceinline__ void warp_fft(Cx<float> (&v)[8], Cx<float>* buf, int j,
                                         const Cx<float>* tw) {
  constexpr int LOG2L = ilog2c(L), NPASS = (LOG2L + 2) / 3;
  constexpr int R = P + 1 == NPASS ? 1 << (LOG2L - (NPASS - 1) * 3) : 8;
  pass_compute<float, L, 8, R, NS, INV>(v, j, tw);
  if constexpr (P + 1 < NPASS) {
    __syncwarp();
    pass_store<float, L, 8, R, NS>(v, buf, j);
    __syncwarp();
    pass_load<float, L, 8>(v, buf, j);
    warp_fft<L, INV, P + 1, NS * R>(v, buf, j, tw);
  }
}

__device__ __forceinline__ uint32_t shared_of(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, Cx<float> v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.re), "f"(v.im)
               : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// One pass over this CTA's lines of L points. src: their points (pitch L + 1); dst[m]: where
// component c of point j + m L/8 of this line goes (shared::cluster addresses). LINES: lines of
// the CTA, the bound of the debug build's index checks (no code otherwise).
template <int L, int SIGMA, int LINES>
__device__ __forceinline__ void small_pass(const Q4<float>* src, const uint32_t (&dst)[8],
                                           Cx<float>* fft, int line, int j, int c,
                                           const float* beta, const Q4<float>* mult,
                                           const Cx<float>* tw, const Q4<float>* u_load,
                                           const Q4<float>* u_store) {
  constexpr int J = L / 8;
  const float sg = c ? -1.f : 1.f;
  auto at = [&](int i) { return dbg_at(line * L + i, (size_t)LINES * L); };
  const Cx<float>* in = reinterpret_cast<const Cx<float>*>(src) + c;
  Cx<float>* buf = fft + line * SGeo<L>::STRIDE + c * SGeo<L>::COMP;
  Cx<float> v[8], p[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int i = j + m * J;
    Cx<float> own = in[2 * dbg_at(line * (L + 1) + i, (size_t)LINES * (L + 1))];
    Cx<float> oth = shfl_pair(own);
    if (u_load) {
      own = apply_u_row(ldg_q4(u_load + at(i)), own, oth, c);
      oth = shfl_pair(own);
    }
    p[m] = own;
    const Cx<float> p1 = c ? oth : own, p2 = c ? own : oth;
    if constexpr (SIGMA == 0) v[m] = {p1.re + sg * p2.re, p1.im + sg * p2.im};
    else v[m] = {p1.re + sg * p2.im, p1.im - sg * p2.re};
  }
  warp_fft<L, false>(v, buf, j, tw);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const Q4<float> q = mult[dbg_at(j + m * J, (size_t)L)];
    const float vr = v[m].re, vi = v[m].im;
    const float sh = -sg * q.z, sl = -sg * q.w;
    v[m] = {fma_t(q.x, vr, fma_t(-sh, vi, fma_t(-sl, vi, q.y * vr))),
            fma_t(q.x, vi, fma_t(sh, vr, fma_t(sl, vr, q.y * vi)))};
  }
  warp_fft<L, true>(v, buf, j, tw);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int i = j + m * J;
    const Cx<float> oth = shfl_pair(v[m]);
    const Cx<float> dp = c ? oth : v[m], dm = c ? v[m] : oth;
    Cx<float> d;
    if (c == 0) d = cadd_p(dp, dm);
    else d = SIGMA == 0 ? csub_p(dp, dm) : mul_i(csub_p(dp, dm));
    const float bm1 = beta[at(i)];
    Cx<float> o = cfma_p(bm1, d, cadd_p(p[m], d));
    if (u_store) o = apply_u_row(u_store[at(i)], o, shfl_pair(o), c);
    st_remote(dst[m], o);
  }
}

// steps of a call: U before the first (lead), U after the last (trail), U^2 between.
template <int LX, int LY, int NC>
__global__ void __launch_bounds__(SPlan<LX, LY, NC>::THREADS)
    k_small_steps(const SmallStepArgs a, int n, int lead, int trail) {
  using S = SPlan<LX, LY, NC>;
  extern __shared__ __align__(16) unsigned char sm[];
  Q4<float>* sa = reinterpret_cast<Q4<float>*>(sm + S::A);
  Q4<float>* sb = reinterpret_cast<Q4<float>*>(sm + S::B);
  Q4<float>* su2 = reinterpret_cast<Q4<float>*>(sm + S::U2);
  Q4<float>* smx = reinterpret_cast<Q4<float>*>(sm + S::MX);
  Q4<float>* smy = reinterpret_cast<Q4<float>*>(sm + S::MY);
  float* sb1 = reinterpret_cast<float*>(sm + S::B1);
  float* sb2 = reinterpret_cast<float*>(sm + S::B2);
  Cx<float>* fft = reinterpret_cast<Cx<float>*>(sm + S::FFT);
  const int tid = threadIdx.x, rank = (int)cooperative_groups::this_cluster().block_rank();
  const size_t row0 = (size_t)rank * S::ROWS * LX, col0 = (size_t)rank * S::COLS * LY;
  auto gz = [&](size_t i) { return dbg_at(i, (size_t)LX * LY); };  // points of the global arrays
  pdl_wait();
  pdl_launch_next();
  for (int k = tid; k < S::ROWS * LX; k += S::THREADS) {
    sa[dbg_at((k / LX) * S::PX + k % LX, S::ROWS * S::PX)] = a.psi[gz(row0 + k)];
    sb1[k] = a.beta1[gz(row0 + k)];
  }
  for (int k = tid; k < S::COLS * LY; k += S::THREADS) {
    sb2[k] = a.beta2[gz(col0 + k)];
    if (a.u2_t) su2[k] = a.u2_t[gz(col0 + k)];
  }
  for (int k = tid; k < LX; k += S::THREADS) smx[k] = a.mult_x[k];
  for (int k = tid; k < LY; k += S::THREADS) smy[k] = a.mult_y[k];

  // this thread's line, point index and component in the two passes, and where its points go
  constexpr int TX = LX / 4, TY = LY / 4;
  const int lx = tid / TX, jx = (tid % TX) >> 1, ly = tid / TY, jy = (tid % TY) >> 1;
  const int c = tid & 1;
  uint32_t dx[8], dy[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int ix = jx + m * (LX / 8);  // x index of the point: column ix % COLS of CTA ix / COLS
    dx[m] = shared_of(smem_u32(sb + dbg_at((ix % S::COLS) * S::PY + rank * S::ROWS + lx,
                                           S::COLS * S::PY)) + 8 * c,
                      (int)dbg_at(ix / S::COLS, NC));
    const int iy = jy + m * (LY / 8);  // y index: row iy % ROWS of CTA iy / ROWS
    dy[m] = shared_of(smem_u32(sa + dbg_at((iy % S::ROWS) * S::PX + rank * S::COLS + ly,
                                           S::ROWS * S::PX)) + 8 * c,
                      (int)dbg_at(iy / S::ROWS, NC));
  }
  cluster_barrier();  // every CTA of the cluster runs, its buffers are filled
  for (int s = 0; s < n; ++s) {
    small_pass<LX, 0, S::ROWS>(sa, dx, fft, lx, jx, c, sb1, smx, a.tw_x,
                      s == 0 && lead && a.u_n ? a.u_n + row0 : nullptr, nullptr);
    cluster_barrier();
    const Q4<float>* us = a.u2_t ? su2 : nullptr;
    if (s + 1 == n && trail && a.u_t) us = a.u_t + col0;
    small_pass<LY, 1, S::COLS>(sb, dy, fft, ly, jy, c, sb2, smy, a.tw_y, nullptr, us);
    cluster_barrier();
  }
  for (int k = tid; k < S::ROWS * LX; k += S::THREADS)
    a.psi[gz(row0 + k)] = sa[dbg_at((k / LX) * S::PX + k % LX, S::ROWS * S::PX)];
}

template <int LX, int LY, int NC>
cudaError_t launch_as(const SmallStepArgs& a, int n, int lead, int trail, cudaStream_t st) {
  using S = SPlan<LX, LY, NC>;
  auto kern = k_small_steps<LX, LY, NC>;
  static int usable[64] = {0};  // per device: 1 a cluster of NC fits, -1 it does not
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!usable[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    if (e == cudaSuccess && NC > 8)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(NC);
    cfg.blockDim = dim3(S::THREADS);
    cfg.dynamicSmemBytes = S::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = NC;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int fit = 0;
    e = cudaOccupancyMaxActiveClusters(&fit, kern, &cfg);
    if (e != cudaSuccess) return e;
    usable[dev] = fit > 0 ? 1 : -1;
  }
  if (usable[dev] < 0) return cudaErrorNotSupported;
  return launch_pdl(kern, dim3(NC), dim3(S::THREADS), S::SMEM, st, true, NC, a, n, lead, trail);
}

}  // namespace

int dgb_debug_flag_small() { return dgb_take_debug_flag(); }

bool small_steps_grid(int nx, int ny) {
  return (nx == 64 || nx == 128) && (ny == 64 || ny == 128);
}

cudaError_t launch_small_steps(const SmallStepArgs& a, int nx, int ny, int n, bool lead,
                               bool trail, cudaStream_t st) {
  if (!small_steps_grid(nx, ny) || n < 1) return cudaErrorInvalidValue;
  if (nx == 64 && ny == 64) return launch_as<64, 64, 16>(a, n, lead, trail, st);
  if (nx == 64) return launch_as<64, 128, 16>(a, n, lead, trail, st);
  if (ny == 64) return launch_as<128, 64, 16>(a, n, lead, trail, st);
  return launch_as<128, 128, 16>(a, n, lead, trail, st);
}

}  // namespace dgb
