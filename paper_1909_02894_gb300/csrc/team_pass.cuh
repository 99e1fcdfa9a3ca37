// Radix-16 line pass for complex64 lines of 256..4096 points (step mode).
//
// A team of T = L/16 threads transforms one line; each thread holds 16 points of both
// eigencomponents in registers, so the points it loads are the points it finishes, and the
// two components share every twiddle, multiplier and barrier. The FFT is a decimation in
// frequency over n = j + T m: DFT-16 over m (registers) -> k0, twiddle W_L^(j k0), team
// exchange; the block of T elements of each k0 then belongs to R2 = L/256 consecutive
// threads of one warp (u = 0..R2-1 holds n' = u + R2 r): DFT-16 over r -> k1, twiddle
// W_T^(u k1), exchange inside the block (no barrier beyond the warp's), DFT-R2 over u ->
// k2. Frequency k = k0 + 16 k1 + 256 k2 is multiplied from a table in exactly that order
// (team_perm), and the inverse runs the same steps backwards with conjugate twiddles. Each
// exchange writes only slots that its own thread (team exchange) or its own block (block
// exchange) has read last, so a line needs two team barriers for its exchanges.
//
// The spinor rows of the next line land in the exchange buffer itself (bulk copy, one
// mbarrier) while the current line's last DFT and epilogue run; the values the epilogue
// needs again are parked in tensor memory. PAIR: a group runs two adjacent lines one after
// the other, keeps the first one's results in tensor memory and writes both lines' points
// together as whole 32-byte sectors straight from registers; otherwise the CTA's LPC lines
// are staged in shared memory and leave in segments of LPC points.
//
// What bounds it, by ncu (profiles/line_pass_team_*.md): at 4096^2 the shared-memory/L1 data pipe
// (exchanges: 128 B per point) and instruction issue, both about half busy, with 16 warps of 128
// registers per SM; at 1024^2, whose 512 pairs of lines make 256 CTAs, latency: 6.4 warps per SM,
// issue 23..25 % and data pipe 31..35 % busy.
// Measured per step of two passes, against the design before it (one 1024-thread CTA per SM
// in radix 8 with one eigencomponent per thread, three exchanges per FFT): 4096^2 0.507 ->
// 0.370 ms, 2048^2 0.165 -> 0.085, 1024^2 0.0439 -> 0.0291 (all three with programmatic
// dependent launch, 0.0045 of it), and with output kinds as template parameters 0.348, 0.085 and
// 0.0282. What mattered, 4096^2: both components per thread and
// radix 16 (34 K -> 23 K warp instructions per 4096 points); coefficient loads in batches
// of four points (0.58 -> 0.48 ms) and stores without a place in L1 (0.44 -> 0.40: the
// tables stay there); prefetch of the coefficients into L2 by the threads instead of bulk
// prefetches (0.473 -> 0.441); sigma as a template parameter (0.392 -> 0.372: the branches
// missed the instruction cache); 32-byte instead of two 16-byte stores (0.62 -> 0.58).
// Tried and not kept: multiplier table and twiddles in shared memory with one CTA of
// independent groups per SM (no faster at 4096^2, 5 % slower at 2048^2), requesting the
// next four points' coefficients early (spills; even).
//
// Every wait on an mbarrier is bounded: if one runs out, the group records an error code in
// *err, stops, waits (bounded) for the copy it issued and leaves.
#pragma once
#include "line_pass.cuh"

namespace dgb {

constexpr uint64_t kWaitNs = 1500000000ull;  // 1.5 s: a copy of 64 KB takes microseconds
constexpr int kErrTimeout = 1;

// Geometry of one line: T threads, blocks of R2 of them, exchange slots.
template <int L>
struct TLine {
  static constexpr int T = L / 16;       // threads of a team
  static constexpr int R2 = L / 256;     // last radix, threads of a block
  static constexpr int NB = 16 / R2;     // last-radix butterflies per thread
  // Slots (8 bytes) between blocks and between the rows of a block: both exchanges touch 16
  // different 8-byte banks per half-warp when BS = R2 mod 16 and RS = R2 + 1.
  static constexpr int BS = R2 == 16 ? 272 : R2 == 8 ? 152 : R2 == 4 ? 84 : R2 == 2 ? 50 : 17;
  static constexpr int RS = R2 + 1;
  static constexpr int COMP = 16 * BS;              // slots of one component of a line
  static constexpr size_t LINE_BYTES = 2 * (size_t)COMP * 8;
  static_assert(BS % 16 == R2 % 16 && BS >= 16 * RS - (R2 == 1 ? 15 : 0), "exchange layout");
  static_assert(LINE_BYTES >= (size_t)L * 16, "landing rows fit the exchange buffer");
};

// LPC teams per CTA. PAIR: groups of GT threads (a team, or the two teams of a warp) work
// independently on their own units and mbarriers; otherwise the CTA is one group.
template <int L, int LPC_, bool PAIR>
struct TGeo : TLine<L> {
  using TL = TLine<L>;
  static constexpr int T = TL::T, R2 = TL::R2;
  static constexpr int LPC = LPC_;       // teams of a CTA
  static constexpr int THREADS = LPC * T;
  static constexpr int GT = PAIR ? (T > 32 ? T : 32) : THREADS;  // threads of a group
  static constexpr int GROUPS = THREADS / GT;
  static constexpr int LG = GT / T;                // lines a group runs at once
  static constexpr int LPU = LG * (PAIR ? 2 : 1);  // lines of a work unit
  static constexpr int SPITCH = L + (LPC > 1 ? 8 / LPC : 0);  // staging rows (points)
  static constexpr size_t XBYTES = LPC * TL::LINE_BYTES;
  static constexpr size_t STAGE = PAIR ? 0 : (size_t)LPC * SPITCH * 16;
  static constexpr size_t OFF_BAR = ((XBYTES > STAGE ? XBYTES : STAGE) + 15) / 16 * 16;
  // per group: an mbarrier and a failure flag; then the tensor-memory address
  static constexpr size_t OFF_SLOT = OFF_BAR + 16 * GROUPS;
  static constexpr size_t OFF_TW2 = OFF_SLOT + 16;
  static constexpr size_t SMEM = OFF_TW2 + 15 * R2 * 8;
  // resident CTAs: 512 threads of 128 registers; at most 512 columns of tensor memory
  static constexpr int MINB = PAIR ? 512 / THREADS : THREADS >= 64 ? 512 / THREADS : 8;
  static constexpr uint32_t PARK = PAIR ? 128 : 64;  // tensor-memory columns per thread
  static constexpr uint32_t TCOLS = PARK * (THREADS > 128 ? THREADS / 128 : 1);
  static_assert(THREADS % 32 == 0 && (THREADS <= 128 || THREADS % 128 == 0), "lane quarters");
  static_assert(SMEM <= 227 * 1024 && (SMEM + 1024) * MINB <= 228 * 1024, "resident CTAs");
  static_assert(TCOLS * MINB <= 512, "tensor memory of the resident CTAs");
};

template <int T, int LPC>
__device__ __forceinline__ void team_sync(int lt) {
  if constexpr (T <= 32) __syncwarp();
  else if constexpr (LPC == 1) __syncthreads();
  else named_barrier(1 + lt, T);
}

// Coefficients of a line (b - 1, U) are read once per pass: loaded without a place in L1,
// which keeps the multiplier and twiddle tables there.
__device__ __forceinline__ Q4<float> ld_stream_q4(const Q4<float>* p) {
  Q4<float> v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
// The same through the coherent path, for arrays that an earlier kernel of the chain writes (see
// launch_pdl: this kernel may be resident while that one still runs, so its data is not
// read-only for this kernel's lifetime, which ld.global.nc asks for).
__device__ __forceinline__ Q4<float> ld_chain_q4(const Q4<float>* p) {
  Q4<float> v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ float ld_stream(const float* p) {
  float v;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
// A pointer of a batched instance, loaded where it is used (a volatile load is not kept in
// registers across the transforms, which have none to spare).
template <typename P>
__device__ __forceinline__ P* ld_ptr(P* const* p) {
  unsigned long long v;
  asm volatile("ld.global.nc.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return reinterpret_cast<P*>(v);
}
// 32 bytes (two adjacent points) in one store, without a place in L1
__device__ __forceinline__ void st_points2(Q4<float>* dst, const float* a, const float* b) {
  asm volatile("st.global.L1::no_allocate.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(a[0]),
               "f"(a[1]), "f"(a[2]), "f"(a[3]), "f"(b[0]), "f"(b[1]), "f"(b[2]), "f"(b[3])
               : "memory");
}

template <int R2, bool INV>
__device__ __forceinline__ void team_dft_r2(Cx<float> (&v)[16]) {
  if constexpr (R2 == 16) {
    dft16<float, INV, false>(v);
  } else if constexpr (R2 > 1) {
#pragma unroll
    for (int q = 0; q < 16 / R2; ++q) {
      Cx<float> x[R2];
#pragma unroll
      for (int t = 0; t < R2; ++t) x[t] = v[q * R2 + t];
      dftR<float, R2, INV>(x);
#pragma unroll
      for (int t = 0; t < R2; ++t) v[q * R2 + t] = x[t];
    }
  }
}

// rows of a line brought into L2, one request per 128 bytes
template <int L, typename V>
__device__ __forceinline__ void team_prefetch(const V* p, int j) {
  constexpr int STEP = 128 / sizeof(V);
  for (int t = j * STEP; t < L; t += L / 16 * STEP)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + t));
}

// From the loaded points (element m of thread j: point j + T m, both components) through the
// forward FFT, the multiply and the inverse FFT up to its last DFT-16, which the caller runs
// after it has released the exchange buffer. xp: the line's exchange buffer, blk: this
// thread's block in it; tw1, tw2, mt: this thread's twiddles W_L^(j k) (stride T) and
// W_T^(u k) (stride R2, shared memory) and multipliers (stride T). mid runs once, between the
// first exchange's writes and its barrier.
template <int L, int LPC, bool DERIV, typename Mid>
__device__ __forceinline__ void team_transform(Cx<float> (&vp)[16], Cx<float> (&vm)[16],
                                               Cx<float>* xp, Cx<float>* blk,
                                               const Cx<float>* tw1, const Cx<float>* tw2,
                                               const Q4<float>* mt, int lt, int j, int u, Mid mid) {
  using G = TLine<L>;
  constexpr int T = G::T, R2 = G::R2, NB = G::NB, BS = G::BS, RS = G::RS;
  // exchange slots of the line and from the block's first one (debug index checks)
  auto xz = [&](int i) { return (int)dbg_at(i, (size_t)2 * G::COMP); };
  auto bz = [&](int i) { return (int)dbg_at(i, (size_t)2 * G::COMP - (j / R2) * BS); };
  dft16<float, false, false>(vp);
  dft16<float, false, false>(vm);
  team_sync<T, LPC>(lt);  // the landing rows have been read
  {
    const Cx<float>* tw = tw1;
    xp[xz(j)] = vp[0];
    xp[xz(G::COMP + j)] = vm[0];
#pragma unroll
    for (int k = 1; k < 16; ++k) {
      const Cx<float> w = ldg_cx(tw + (k - 1) * T);
      xp[xz(k * BS + j)] = cmul(vp[k], w);
      xp[xz(G::COMP + k * BS + j)] = cmul(vm[k], w);
    }
  }
  mid();
  team_sync<T, LPC>(lt);
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    vp[r] = blk[bz(u + R2 * r)];
    vm[r] = blk[bz(G::COMP + u + R2 * r)];
  }
  dft16<float, false, false>(vp);
  dft16<float, false, false>(vm);
  if constexpr (R2 > 1) {
    const Cx<float>* tw = tw2;
    __syncwarp();  // the block's threads have read it
    blk[bz(u)] = vp[0];
    blk[bz(G::COMP + u)] = vm[0];
#pragma unroll
    for (int k = 1; k < 16; ++k) {
      const Cx<float> w = tw[(k - 1) * R2];
      blk[bz(k * RS + u)] = cmul(vp[k], w);
      blk[bz(G::COMP + k * RS + u)] = cmul(vm[k], w);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int t = 0; t < R2; ++t) {
        vp[q * R2 + t] = blk[bz((u + R2 * q) * RS + t)];
        vm[q * R2 + t] = blk[bz(G::COMP + (u + R2 * q) * RS + t)];
      }
    team_dft_r2<R2, false>(vp);
    team_dft_r2<R2, false>(vm);
  }
  // k-space multiply. Step: eigenvalue +1 by (cos - 1) - i sin, -1 by (cos - 1) + i sin;
  // derivative: both components by i xi
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const Q4<float> q = ldg_q4(mt + e * T);
    {
      const float vr = vp[e].re, vi = vp[e].im;
      if constexpr (DERIV)
        vp[e] = {-(q.z * vi + q.w * vi), q.z * vr + q.w * vr};
      else
        vp[e] = {q.x * vr + ((q.y * vr + q.w * vi) + q.z * vi),
                 q.x * vi + ((q.y * vi - q.w * vr) - q.z * vr)};
    }
    {
      const float vr = vm[e].re, vi = vm[e].im;
      if constexpr (DERIV)
        vm[e] = {-(q.z * vi + q.w * vi), q.z * vr + q.w * vr};
      else
        vm[e] = {q.x * vr + ((q.y * vr - q.w * vi) - q.z * vi),
                 q.x * vi + ((q.y * vi + q.w * vr) + q.z * vr)};
    }
  }
  if constexpr (R2 > 1) {
    team_dft_r2<R2, true>(vp);
    team_dft_r2<R2, true>(vm);
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int t = 0; t < R2; ++t) {
        blk[bz((u + R2 * q) * RS + t)] = vp[q * R2 + t];
        blk[bz(G::COMP + (u + R2 * q) * RS + t)] = vm[q * R2 + t];
      }
    __syncwarp();
    const Cx<float>* tw = tw2;
    vp[0] = blk[bz(u)];
    vm[0] = blk[bz(G::COMP + u)];
#pragma unroll
    for (int k = 1; k < 16; ++k) {
      const Cx<float> w = tw[(k - 1) * R2];
      vp[k] = cmulc(blk[bz(k * RS + u)], w);
      vm[k] = cmulc(blk[bz(G::COMP + k * RS + u)], w);
    }
    __syncwarp();  // the block's threads have read it
  }
  dft16<float, true, false>(vp);
  dft16<float, true, false>(vm);
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    blk[bz(u + R2 * r)] = vp[r];
    blk[bz(G::COMP + u + R2 * r)] = vm[r];
  }
  team_sync<T, LPC>(lt);
  {
    const Cx<float>* tw = tw1;
    asm volatile("" : "+l"(tw));
    vp[0] = xp[xz(j)];
    vm[0] = xp[xz(G::COMP + j)];
#pragma unroll
    for (int k = 1; k < 16; ++k) {
      const Cx<float> w = ldg_cx(tw + (k - 1) * T);
      vp[k] = cmulc(xp[xz(k * BS + j)], w);
      vm[k] = cmulc(xp[xz(G::COMP + k * BS + j)], w);
    }
  }
}

// What a step pass does with its results. Kinds and sigma are template parameters since the
// kernel's speed depends on its code size (the branches of one general kernel, taken or not,
// cost 4..6 % in instruction-cache misses at 1024^2 and 4096^2).
enum TeamOut {
  TEAM_PLAIN = 0,  // transposed store, no U (x passes; sigma_x: U on load if u_load is set)
  TEAM_U = 1,      // transposed store after U (y passes; batches: if the instance has one)
  TEAM_UG = 2,     // transposed store after a general U (static potentials)
  TEAM_ROWS = 3    // rows back in the input's layout, after U or a general U if set
};

template <int L, int LPC, bool PAIR, bool BATCH, int SIGMA, int OUT>
__global__ void __launch_bounds__(TGeo<L, LPC, PAIR>::THREADS, TGeo<L, LPC, PAIR>::MINB)
    line_pass_team(const LinePassArgs<float> a0, int n_units, int* __restrict__ err) {
  using G = TGeo<L, LPC, PAIR>;
  constexpr int T = G::T, R2 = G::R2, BS = G::BS;
  constexpr bool U_OUT = OUT == TEAM_U || OUT == TEAM_ROWS;
  constexpr bool UG_OUT = OUT == TEAM_UG || OUT == TEAM_ROWS;
  extern __shared__ __align__(128) unsigned char tsm[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int lt = tid / T, j = tid - lt * T;
  const int u = j % R2;
  const int grp = tid / G::GT, lg = lt - grp * G::LG;  // group, line within it
  uint64_t* bar = reinterpret_cast<uint64_t*>(tsm + G::OFF_BAR + 16 * grp);
  int* bad = reinterpret_cast<int*>(tsm + G::OFF_BAR + 16 * grp + 8);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tsm + G::OFF_SLOT);
  unsigned char* zone = tsm + lt * G::LINE_BYTES;
  Cx<float>* xp = reinterpret_cast<Cx<float>*>(zone);  // + component, - component at xp + COMP
  Cx<float>* blk = xp + (j / R2) * BS;
  Q4<float>* land = reinterpret_cast<Q4<float>*>(zone);
  const bool leader = tid == grp * G::GT;

  pdl_wait();
  const int upi = a0.n_lines / G::LPU;  // units of an instance
  // index checks of the debug build (no code otherwise): landing rows, staging, points of the
  // global arrays
  auto lz = [&](int i) { return (int)dbg_at(i, (size_t)L); };
  auto sz = [&](int i) { return (int)dbg_at(i, (size_t)LPC * G::SPITCH); };
  auto gz = [&](size_t i) { return dbg_at(i, (size_t)a0.n_lines * L); };
  if constexpr (BATCH) n_units = *a0.n_inst * upi;
  auto group_sync = [&]() {
    if constexpr (G::GT == 32) __syncwarp();
    else if constexpr (G::GROUPS == 1) __syncthreads();
    else named_barrier(1 + grp, G::GT);
  };
  // leader: request the rows of sub-line h of a unit
  auto issue = [&](int unit, int h) {
    LinePassArgs<float> x = a0;
    if constexpr (BATCH) {
      bind_instance(x, unit / upi);
      unit = unit % upi;
    }
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (uint32_t)(G::LG * L * 16) + x.test_extra_tx);
#pragma unroll 1
    for (int l = 0; l < G::LG; ++l) {
      const size_t first = (size_t)(unit * G::LPU + (PAIR ? 2 * l + h : l)) * L;
      bulk_copy_g2s(tsm + (grp * G::LG + l) * G::LINE_BYTES, x.in + first, L * 16, bar);
    }
  };

  Cx<float>* tw2s = reinterpret_cast<Cx<float>*>(tsm + G::OFF_TW2);
  if (leader) {
    mbar_init(bar, 1);
    *bad = 0;
    fence_mbar_init();
  }
  int unit = blockIdx.x + gridDim.x * grp;
  if (leader && unit < n_units) issue(unit, 0);
  if (warp == 0) tmem_alloc(tslot, G::TCOLS);
  for (int t = tid; t < 15 * R2; t += G::THREADS) tw2s[t] = ldg_cx(a0.tw + 15 * T + t);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  // only now: the next kernel's CTAs take tensor memory when they start and keep it while they
  // wait for this kernel, so every CTA of this one must hold its own first
  pdl_launch_next();
  const uint32_t tbase = *tslot;
  const uint32_t tpark =
      tbase + ((32u * (uint32_t)(warp & 3)) << 16) + G::PARK * (uint32_t)(warp >> 2);

  bool failed = false;
  uint32_t par = 0;
  int h = 0;
  while (unit < n_units) {
    const InstPtrs<float>* ip = BATCH ? a0.inst + unit / upi : nullptr;  // the unit's instance
    const int ul = BATCH ? unit % upi : unit;
    const int line = ul * G::LPU + (PAIR ? 2 * lg + h : lg);
    const size_t row = (size_t)line * L;
    Cx<float> vp[16], vm[16];
    const bool ok = mbar_wait_bounded(bar, par, kWaitNs);
    par ^= 1u;
    if constexpr (SIGMA == 0 && OUT == TEAM_PLAIN) {
      const Q4<float>* u_load = BATCH ? ld_ptr(&ip->u_load) : a0.u_load;
      if (u_load) {  // first pass of a call: U applied to the landed points in place
#pragma unroll 4
        for (int m = 0; m < 16; ++m)
          land[lz(j + T * m)] =
              apply_u(ld_stream_q4(u_load + gz(row + j + T * m)), land[lz(j + T * m)]);
      }
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      float pk[16];
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) {
        const int m = 4 * g + mm;
        const Q4<float> p = land[lz(j + T * m)];
        pk[4 * mm] = p.x;
        pk[4 * mm + 1] = p.y;
        pk[4 * mm + 2] = p.z;
        pk[4 * mm + 3] = p.w;
        if constexpr (SIGMA == 0) {
          vp[m] = cadd_p(Cx<float>{p.x, p.y}, Cx<float>{p.z, p.w});
          vm[m] = csub_p(Cx<float>{p.x, p.y}, Cx<float>{p.z, p.w});
        } else {
          vp[m] = {p.x + p.w, p.y - p.z};
          vm[m] = {p.x - p.w, p.y + p.z};
        }
      }
      tmem_st16(tpark + (uint32_t)((PAIR ? 64 * h : 0) + 16 * g), pk);
    }
    const Q4<float>* mult = BATCH ? ld_ptr(&ip->mult_perm) : a0.mult_perm;
    team_transform<L, LPC, false>(vp, vm, xp, blk, a0.tw + j, tw2s + u, mult + j, lt, j, u, [&]() {
      // the line's coefficients into L2, a line's transforms ahead of their use (bulk
      // prefetches queue with the landing copies and were slower)
      team_prefetch<L>((BATCH ? ld_ptr(&ip->beta) : a0.beta) + row, j);
      if constexpr (U_OUT) {
        const Q4<float>* us = BATCH ? ld_ptr(&ip->u_store) : a0.u_store;
        if (us) team_prefetch<L>(us + row, j);
      }
      if (UG_OUT && a0.ug_store) {
        team_prefetch<L>(a0.ug_store + 2 * row, j);
        team_prefetch<L>(a0.ug_store + 2 * row + L, j);
      }
    });
    // the exchange buffer is free: the next rows may land in it
    if (!ok) *bad = 1;
    group_sync();
    if (*bad) {
      failed = true;
      break;
    }
    const int next = unit + (int)gridDim.x * G::GROUPS;
    if constexpr (PAIR) {
      if (leader) {
        if (h == 0) issue(unit, 1);
        else if (next < n_units) issue(next, 0);
      }
    }
    dft16<float, true, false>(vp);
    dft16<float, true, false>(vm);
    tmem_wait_st();
    // ---- epilogue: psi + D + (b - 1) D, U; coefficients in batches of four points
    const float* beta = BATCH ? ld_ptr(&ip->beta) : a0.beta;
    const Q4<float>* u_store = !U_OUT ? nullptr : BATCH ? ld_ptr(&ip->u_store) : a0.u_store;
    Q4<float>* out = BATCH ? ld_ptr(&ip->out) : a0.out;
    const bool has_u = U_OUT && ((!BATCH && OUT == TEAM_U) || u_store != nullptr);
    // transposed store of the pair: row j + T m of the output (the opaque step keeps the
    // compiler from holding sixteen row offsets across the loop)
    size_t dstep = (size_t)T * a0.n_lines;
    asm volatile("" : "+l"(dstep));
    Q4<float>* dst = out + (size_t)j * a0.n_lines + (line - 1);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const size_t g0 = row + j + T * 4 * g;
      float pk[16], bc[4];
      Q4<float> uc[4];
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) bc[mm] = ld_stream(beta + gz(g0 + T * mm));
      if constexpr (U_OUT) {
        if (has_u) {
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) uc[mm] = ld_stream_q4(u_store + gz(g0 + T * mm));
        }
      }
      tmem_ld16(tpark + (uint32_t)((PAIR ? 64 * h : 0) + 16 * g), pk);
      tmem_wait_ld_regs(pk);
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) {
        const int m = 4 * g + mm;
        const Cx<float> d1 = cadd_p(vp[m], vm[m]), dd = csub_p(vp[m], vm[m]);
        const float bm1 = bc[mm];
        const Cx<float> o1 = cfma_p(bm1, d1, cadd_p(Cx<float>{pk[4 * mm], pk[4 * mm + 1]}, d1));
        Cx<float> o2;
        if constexpr (SIGMA == 0) {
          o2 = cfma_p(bm1, dd, cadd_p(Cx<float>{pk[4 * mm + 2], pk[4 * mm + 3]}, dd));
        } else {
          const Cx<float> d2 = mul_i(dd);
          o2 = {(pk[4 * mm + 2] + d2.re) + bm1 * d2.re, (pk[4 * mm + 3] + d2.im) + bm1 * d2.im};
        }
        pk[4 * mm] = o1.re;
        pk[4 * mm + 1] = o1.im;
        pk[4 * mm + 2] = o2.re;
        pk[4 * mm + 3] = o2.im;
      }
      if constexpr (U_OUT) {
        if (has_u) {
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            const Q4<float> o =
                apply_u(uc[mm], Q4<float>{pk[4 * mm], pk[4 * mm + 1], pk[4 * mm + 2], pk[4 * mm + 3]});
            pk[4 * mm] = o.x;
            pk[4 * mm + 1] = o.y;
            pk[4 * mm + 2] = o.z;
            pk[4 * mm + 3] = o.w;
          }
        }
      }
      if constexpr (UG_OUT) {
        if (OUT == TEAM_UG || a0.ug_store) {  // static potentials
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            const Q4<float>* ug = a0.ug_store + 2 * gz(g0 + T * mm);
            const Q4<float> o = apply_u_general(
                ld_stream_q4(ug), ld_stream_q4(ug + 1),
                Q4<float>{pk[4 * mm], pk[4 * mm + 1], pk[4 * mm + 2], pk[4 * mm + 3]});
            pk[4 * mm] = o.x;
            pk[4 * mm + 1] = o.y;
            pk[4 * mm + 2] = o.z;
            pk[4 * mm + 3] = o.w;
          }
        }
      }
      if constexpr (OUT == TEAM_ROWS) {
#pragma unroll
        for (int mm = 0; mm < 4; ++mm)
          out[gz(g0 + T * mm)] = {pk[4 * mm], pk[4 * mm + 1], pk[4 * mm + 2], pk[4 * mm + 3]};
      } else if constexpr (!PAIR) {
#pragma unroll
        for (int mm = 0; mm < 4; ++mm)
          reinterpret_cast<Q4<float>*>(tsm)[sz(lt * G::SPITCH + j + T * (4 * g + mm))] = {
              pk[4 * mm], pk[4 * mm + 1], pk[4 * mm + 2], pk[4 * mm + 3]};
      }
      if constexpr (PAIR && OUT != TEAM_ROWS) {
        if (h == 0) {
          tmem_st16(tpark + (uint32_t)(16 * g), pk);
        } else {
          float pa[16];
          tmem_ld16(tpark + (uint32_t)(16 * g), pa);
          tmem_wait_ld_regs(pa);
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            if (dbg_in((size_t)(dst - out) + 1, (size_t)a0.n_lines * L))
              st_points2(dst, pa + 4 * mm, pk + 4 * mm);
            dst += dstep;
          }
        }
      }
    }
    if constexpr (PAIR) {
      if (h == 0) {
        h = 1;
      } else {
        h = 0;
        unit = next;
      }
    } else {
      __syncthreads();
      if constexpr (OUT != TEAM_ROWS) {
        const Q4<float>* st = reinterpret_cast<const Q4<float>*>(tsm);
        const int g = tid % LPC, i0 = tid / LPC;
        Q4<float>* dst = out + (size_t)i0 * a0.n_lines + (ul * G::LPU + g);
        constexpr int RPI = G::THREADS / LPC;
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (dbg_in((size_t)(i0 + q * RPI) * a0.n_lines + ul * G::LPU + g, (size_t)a0.n_lines * L))
            dst[(size_t)(q * RPI) * a0.n_lines] = st[sz(g * G::SPITCH + i0 + q * RPI)];
        __syncthreads();
      }
      unit = next;
      if (leader && unit < n_units) issue(unit, 0);
    }
  }
  if (failed && leader) {
    atomicExch(err, kErrTimeout);
    mbar_wait_bounded(bar, par ^ 1u, kWaitNs);  // the copies in flight
  }
  tmem_wait_st();
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(tbase, G::TCOLS);
}

}  // namespace dgb
