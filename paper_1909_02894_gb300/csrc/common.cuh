// Shared device types and helpers for the Scheme II kernels (sm_103a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

// Debug builds (nvcc -DDIRAC_DEBUG=1, see DIRAC_NVCC_EXTRA) check the index of each
// memory access of the line passes against its buffer: a failed check sets this
// translation unit's flag and the access is skipped (a load gives zero). Release builds
// compile the checks away.
#ifndef DIRAC_DEBUG
#define DIRAC_DEBUG 0
#endif

namespace dgb {

#if DIRAC_DEBUG
static __device__ int g_dbg_bounds = 0;
#endif
// Reads and clears this translation unit's flag (always 0 in release builds).
inline static int dgb_take_debug_flag() {
#if DIRAC_DEBUG
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_dbg_bounds, sizeof(int)) != cudaSuccess) return 1;
  if (v) {
    const int z = 0;
    cudaMemcpyToSymbol(g_dbg_bounds, &z, sizeof(int));
  }
  return v;
#else
  return 0;
#endif
}
// true when idx < bound (always, in release builds)
__device__ __forceinline__ bool dbg_in(size_t idx, size_t bound) {
#if DIRAC_DEBUG
  if (idx >= bound) {
    atomicExch(&g_dbg_bounds, 1);
    return false;
  }
#endif
  return true;
}

// idx, or 0 when a debug build finds it out of bounds (a harmless slot of the same array)
__device__ __forceinline__ size_t dbg_at(size_t idx, size_t bound) {
  return dbg_in(idx, bound) ? idx : 0;
}

// Complex number in registers / shared memory.
template <typename T>
struct __align__(2 * sizeof(T)) Cx {
  T re, im;
};

// Four reals: a spinor point (psi1.re, psi1.im, psi2.re, psi2.im), a half-step matrix
// (c0 - 1, c1, c2, c3), or a k-space multiplier (hi/lo pairs).
template <typename T>
struct __align__(4 * sizeof(T)) Q4 {
  T x, y, z, w;
};

template <typename T>
__device__ __forceinline__ Cx<T> cadd(Cx<T> a, Cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T>
__device__ __forceinline__ Cx<T> csub(Cx<T> a, Cx<T> b) { return {a.re - b.re, a.im - b.im}; }
// a b + c in one rounding. Products are written with it where the compiler could contract
// them in two ways, so that every kernel rounds alike (whole-step launches give the bits of
// separate passes).
__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
template <typename T>
__device__ __forceinline__ Cx<T> cmul(Cx<T> a, Cx<T> b) {
  return {fma_t(a.re, b.re, -(a.im * b.im)), fma_t(a.re, b.im, a.im * b.re)};
}
// a * conj(b)
template <typename T>
__device__ __forceinline__ Cx<T> cmulc(Cx<T> a, Cx<T> b) {
  return {fma_t(a.re, b.re, a.im * b.im), fma_t(a.im, b.re, -(a.re * b.im))};
}
// ---- packed FP32 pairs (sm_100 and later): the (re, im) of a complex64 value in one
// 64-bit register pair, two FP32 operations per instruction, each rounded exactly like its
// scalar counterpart (add/sub/fma.rn.f32x2).
__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk2(unsigned long long r, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a,
                                                         unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long sub_f32x2(unsigned long long a,
                                                         unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a * b + c per lane
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a,
                                                         unsigned long long b,
                                                         unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long pk2(Cx<float> a) { return pk2(a.re, a.im); }
__device__ __forceinline__ Cx<float> upk2(unsigned long long r) {
  Cx<float> a;
  upk2(r, a.re, a.im);
  return a;
}

// a + b and a - b: one packed instruction for complex64, the scalar pair otherwise.
// Building with -DDGB_PACKED_F32X2=0 keeps the scalar form for complex64 too (same results).
#ifndef DGB_PACKED_F32X2
#define DGB_PACKED_F32X2 1
#endif
template <typename T>
__device__ __forceinline__ Cx<T> cadd_p(Cx<T> a, Cx<T> b) { return cadd(a, b); }
template <typename T>
__device__ __forceinline__ Cx<T> csub_p(Cx<T> a, Cx<T> b) { return csub(a, b); }
// s * a + b with the same real s on both parts (a single fma.rn.f32x2 for complex64)
template <typename T>
__device__ __forceinline__ Cx<T> cfma_p(T s, Cx<T> a, Cx<T> b) {
  return {s * a.re + b.re, s * a.im + b.im};
}
#if DGB_PACKED_F32X2
template <>
__device__ __forceinline__ Cx<float> cadd_p<float>(Cx<float> a, Cx<float> b) {
  return upk2(add_f32x2(pk2(a), pk2(b)));
}
template <>
__device__ __forceinline__ Cx<float> csub_p<float>(Cx<float> a, Cx<float> b) {
  return upk2(sub_f32x2(pk2(a), pk2(b)));
}
template <>
__device__ __forceinline__ Cx<float> cfma_p<float>(float s, Cx<float> a, Cx<float> b) {
  return upk2(fma_f32x2(pk2(s, s), pk2(a), pk2(b)));
}
#endif

template <typename T>
__device__ __forceinline__ Cx<T> mul_i(Cx<T> a) { return {-a.im, a.re}; }
template <typename T>
__device__ __forceinline__ Cx<T> mul_mi(Cx<T> a) { return {a.im, -a.re}; }

// psi <- U psi with U = [[c0 + i c3, c1 - i c2], [c1 + i c2, c0 - i c3]] stored as
// u = (c0 - 1, c1, c2, c3): the deviation from the identity is applied and added, so a
// U close to I costs one rounding of psi.
template <typename T>
__device__ __forceinline__ Q4<T> apply_u(Q4<T> u, Q4<T> p) {
  const T ar = p.x, ai = p.y, br = p.z, bi = p.w;
  T d1r = u.x * ar - u.w * ai + u.y * br + u.z * bi;
  T d1i = u.x * ai + u.w * ar + u.y * bi - u.z * br;
  T d2r = u.x * br + u.w * bi + u.y * ar - u.z * ai;
  T d2i = u.x * bi - u.w * br + u.y * ai + u.z * ar;
  return {ar + d1r, ai + d1i, br + d2r, bi + d2i};
}

// psi <- U psi for a general complex U stored as its deviation from I: r0 = (d00, u01), r1 =
// (u10, d11).
template <typename T>
__device__ __forceinline__ Q4<T> apply_u_general(Q4<T> r0, Q4<T> r1, Q4<T> p) {
  // (fused explicitly, as cmul is, so that the kernels of both layouts round alike)
  const T a = p.x, b = p.y, c = p.z, d = p.w;
  return {a + fma_t(-r0.w, d, fma_t(r0.z, c, fma_t(r0.x, a, -(r0.y * b)))),
          b + fma_t(r0.w, c, fma_t(r0.z, d, fma_t(r0.y, a, r0.x * b))),
          c + fma_t(-r1.w, d, fma_t(r1.z, c, fma_t(r1.x, a, -(r1.y * b)))),
          d + fma_t(r1.w, c, fma_t(r1.z, d, fma_t(r1.y, a, r1.x * b)))};
}

}  // namespace dgb

namespace dgb {

// ---- asynchronous bulk copies and mbarriers (sm_90+ PTX), used by the team pass
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Orders this thread's earlier generic-proxy shared-memory accesses before later
// async-proxy operations on the same memory (bulk copies that write it, bulk and tensor
// stores that read it).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// Global -> shared bulk copy (16-B aligned addresses, size a multiple of 16) whose
// completion is counted on the mbarrier.
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after limit_ns nanoseconds of wall time.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}

// Position of frequency k in the multiplier tables of the radix-16 team pass (lines of L =
// 256..4096 points, team_pass.cuh): thread j = R2 k0 + v of the line's L/16 (R2 = L/256)
// holds frequency k0 + 16 (v + R2 q) + 256 k2 in element e = q R2 + k2, and entry e of thread
// j sits at e L/16 + j, so that a warp reads consecutive entries.
__host__ __device__ constexpr int team_perm(int L, int k) {
  return (((k >> 4) & 15) / (L / 256) * (L / 256) + (k >> 8)) * (L / 16) + (k & 15) * (L / 256) +
         ((k >> 4) & 15) % (L / 256);
}
__host__ __device__ constexpr bool team_length(int L) { return L >= 256 && L <= 4096; }

// Programmatic dependent launch: waits until the kernels this one depends on have completed
// and their writes are visible (at once when launched without the attribute), and lets the
// next kernel of the stream be scheduled (it waits here in turn).
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_launch_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---- tensor memory (tcgen05, sm_100a+) used as per-thread parking space. A CTA holds
// `cols` columns x 128 lanes of 32-bit cells; warp w reaches lanes 32 (w % 4) .. + 31
// (its lane quarter) with the 32x32b shapes, one lane per thread.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {  // one warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {  // one warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tmem_fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// 16 consecutive columns of this thread's lane <- r[0..15]
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
      "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
      : "memory");
}
// r[0..15] <- 16 consecutive columns of this thread's lane (complete after a wait)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]),
        "=f"(r[7]), "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]),
        "=f"(r[14]), "=f"(r[15])
      : "r"(taddr)
      : "memory");
}
// Waits for this thread's tensor-memory loads; naming the destination registers as
// operands keeps every use of them after the wait.
__device__ __forceinline__ void tmem_wait_ld_regs(float (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]),
                 "+f"(r[6]), "+f"(r[7]), "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]),
                 "+f"(r[12]), "+f"(r[13]), "+f"(r[14]), "+f"(r[15])::"memory");
}
// Barrier over `count` threads (a multiple of 32) on hardware barrier `id` (1..15).
__device__ __forceinline__ void named_barrier(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

}  // namespace dgb
