// The operator of the unsplit schemes, S = b^1 sigma_x [[d_x]] + b^2 sigma_y [[d_y]], on
// complex64 states whose axes have 256..4096 points, as two passes of the radix-16 team
// transform (team_pass.cuh) in derivative mode:
//   phase 1  rows of the input: S_axis = b^axis sigma_axis d_axis in, written transposed
//            together with a transposed copy of the input;
//   phase 2  rows of that copy: the other axis' term, out = alpha (S_1 + S_2) + gamma base +
//            beta prev, optionally U out, written as rows (the result is then in the
//            transposed layout, where the next application starts) or transposed back.
// Against separate derivative passes, a transpose and a pointwise combine (four launches,
// 208 B of memory traffic per point): two launches and 120 B; a thread holds both
// components of its points, so the 2 x 2 algebra needs no exchange. Bound like the step pass,
// and by the latency of the coefficient and term loads of the epilogue (up to 52 B per point);
// phase 1 stores twice as much (two transposed arrays). Measured with the whole scheme around
// it: Chebyshev of degree 8 at 1024^2 0.52 -> 0.29 ms per step (0.0193 and 0.0275 ms per phase
// under ncu, profiles/unsplit_chebyshev1024.md, against 0.064 for the four launches).
#pragma once
#include "team_pass.cuh"

namespace dgb {

template <int L, int LPC, bool PAIR, int PHASE>
__global__ void __launch_bounds__(TGeo<L, LPC, PAIR>::THREADS, TGeo<L, LPC, PAIR>::MINB)
    line_pass_team_unsplit(const UnsplitArgs a, int n_units) {
  using G = TGeo<L, LPC, PAIR>;
  constexpr int T = G::T, R2 = G::R2, BS = G::BS;
  extern __shared__ __align__(128) unsigned char tsm[];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int lt = tid / T, j = tid - lt * T;
  const int u = j % R2;
  const int grp = tid / G::GT, lg = lt - grp * G::LG;
  uint64_t* bar = reinterpret_cast<uint64_t*>(tsm + G::OFF_BAR + 16 * grp);
  int* bad = reinterpret_cast<int*>(tsm + G::OFF_BAR + 16 * grp + 8);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tsm + G::OFF_SLOT);
  unsigned char* zone = tsm + lt * G::LINE_BYTES;
  Cx<float>* xp = reinterpret_cast<Cx<float>*>(zone);
  Cx<float>* blk = xp + (j / R2) * BS;
  const Q4<float>* land = reinterpret_cast<const Q4<float>*>(zone);
  Cx<float>* tw2s = reinterpret_cast<Cx<float>*>(tsm + G::OFF_TW2);
  const bool leader = tid == grp * G::GT;
  auto lz = [&](int i) { return (int)dbg_at(i, (size_t)L); };
  auto sz = [&](int i) { return (int)dbg_at(i, (size_t)LPC * G::SPITCH); };
  auto gz = [&](size_t i) { return dbg_at(i, (size_t)a.n_lines * L); };
  auto group_sync = [&]() {
    if constexpr (G::GT == 32) __syncwarp();
    else if constexpr (G::GROUPS == 1) __syncthreads();
    else named_barrier(1 + grp, G::GT);
  };
  auto issue = [&](int unit, int h) {
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, (uint32_t)(G::LG * L * 16) + a.test_extra_tx);
#pragma unroll 1
    for (int l = 0; l < G::LG; ++l)
      bulk_copy_g2s(tsm + (grp * G::LG + l) * G::LINE_BYTES,
                    a.in + (size_t)(unit * G::LPU + (PAIR ? 2 * l + h : l)) * L, L * 16, bar);
  };

  if (leader) {
    mbar_init(bar, 1);
    *bad = 0;
    fence_mbar_init();
  }
  if (PAIR && warp == 0) tmem_alloc(tslot, G::TCOLS);
  pdl_wait();
  int unit = blockIdx.x + gridDim.x * grp;
  if (leader && unit < n_units) issue(unit, 0);
  for (int t = tid; t < 15 * R2; t += G::THREADS) tw2s[t] = ldg_cx(a.tw + 15 * T + t);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  // only now: the next kernel's CTAs take tensor memory when they start and keep it while they
  // wait for this kernel, so every CTA of this one must hold its own first
  pdl_launch_next();
  const uint32_t tbase = PAIR ? *tslot : 0;
  const uint32_t tpark =
      tbase + ((32u * (uint32_t)(warp & 3)) << 16) + G::PARK * (uint32_t)(warp >> 2);

  bool failed = false;
  uint32_t par = 0;
  int h = 0;
  while (unit < n_units) {
    const int line = unit * G::LPU + (PAIR ? 2 * lg + h : lg);
    const size_t row = (size_t)line * L;
    size_t dstep = (size_t)T * a.n_lines;  // transposed stores: points T apart
    asm volatile("" : "+l"(dstep));
    const size_t dst0 = (size_t)j * a.n_lines + (line - 1);  // PAIR, h = 1
    Cx<float> v1[16], v2[16];
    const bool ok = mbar_wait_bounded(bar, par, kWaitNs);
    par ^= 1u;
    if constexpr (PHASE == 1 && !PAIR) {
      // the transposed copy, straight from the landed rows
      const int g = tid % LPC, i0 = tid / LPC;
      const Q4<float>* src = reinterpret_cast<const Q4<float>*>(tsm + g * G::LINE_BYTES);
      Q4<float>* dst = a.out_in + (size_t)i0 * a.n_lines + (unit * G::LPU + g);
      constexpr int RPI = G::THREADS / LPC;
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (dbg_in((size_t)(i0 + q * RPI) * a.n_lines + unit * G::LPU + g, (size_t)a.n_lines * L))
          dst[(size_t)(q * RPI) * a.n_lines] = src[lz(i0 + q * RPI)];
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
        v1[m] = {p.x, p.y};
        v2[m] = {p.z, p.w};
      }
      if constexpr (PHASE == 1 && PAIR) {
        // the transposed copy: the first line's points wait in tensor memory for the second's
        if (h == 0) {
          tmem_st16(tpark + (uint32_t)(16 * g), pk);
        } else {
          float pa[16];
          tmem_ld16(tpark + (uint32_t)(16 * g), pa);
          tmem_wait_ld_regs(pa);
          Q4<float>* dst = a.out_in + dst0 + 4 * g * dstep;
#pragma unroll
          for (int mm = 0; mm < 4; ++mm)
            if (dbg_in(dst0 + (4 * g + mm) * dstep + 1, (size_t)a.n_lines * L))
              st_points2(dst + mm * dstep, pa + 4 * mm, pk + 4 * mm);
        }
      }
    }
    if constexpr (PHASE == 1 && !PAIR) __syncthreads();  // other threads read this line's rows
    team_transform<L, LPC, true>(v1, v2, xp, blk, a.tw + j, tw2s + u, a.mult + j, lt, j, u, [&]() {
      team_prefetch<L>(a.beta + row, j);
      if constexpr (PHASE == 2) {
        team_prefetch<L>(a.s_other + row, j);
        if (a.base) team_prefetch<L>(a.base + row, j);
        if (a.prev) team_prefetch<L>(a.prev + row, j);
        if (a.u_store) team_prefetch<L>(a.u_store + row, j);
      }
    });
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
    dft16<float, true, false>(v1);
    dft16<float, true, false>(v2);
    if constexpr (PAIR) tmem_wait_st();
    // where the first line's results wait for the second's
    const uint32_t tres = tpark + (PHASE == 1 ? 64u : 0u);
    const bool rows_out = PHASE == 2 && a.store_normal;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const size_t g0 = row + j + T * 4 * g;
      float o[16], bm1[4];
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) bm1[mm] = ld_stream(a.beta + gz(g0 + T * mm));
      Q4<float> qb[4];
      if constexpr (PHASE == 2) {
        if (a.base) {
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) qb[mm] = ld_chain_q4(a.base + gz(g0 + T * mm));
        }
#pragma unroll
        for (int mm = 0; mm < 4; ++mm) {
          const Q4<float> s = ld_chain_q4(a.s_other + gz(g0 + T * mm));
          o[4 * mm] = s.x;
          o[4 * mm + 1] = s.y;
          o[4 * mm + 2] = s.z;
          o[4 * mm + 3] = s.w;
        }
      }
#pragma unroll
      for (int mm = 0; mm < 4; ++mm) {
        const int m = 4 * g + mm;
        // sigma_x (d1, d2) = (d2, d1), sigma_y (d1, d2) = (-i d2, i d1)
        const Cx<float> t1 = a.axis == 0 ? v2[m] : mul_mi(v2[m]);
        const Cx<float> t2 = a.axis == 0 ? v1[m] : mul_i(v1[m]);
        // b t = t + (b - 1) t
        const Cx<float> s1 = cfma_p(bm1[mm], t1, t1), s2 = cfma_p(bm1[mm], t2, t2);
        if constexpr (PHASE == 1) {
          o[4 * mm] = s1.re;
          o[4 * mm + 1] = s1.im;
          o[4 * mm + 2] = s2.re;
          o[4 * mm + 3] = s2.im;
        } else {
          const float r1 = o[4 * mm] + s1.re, i1 = o[4 * mm + 1] + s1.im;
          const float r2 = o[4 * mm + 2] + s2.re, i2 = o[4 * mm + 3] + s2.im;
          o[4 * mm] = a.ar * r1 - a.ai * i1;
          o[4 * mm + 1] = a.ar * i1 + a.ai * r1;
          o[4 * mm + 2] = a.ar * r2 - a.ai * i2;
          o[4 * mm + 3] = a.ar * i2 + a.ai * r2;
        }
      }
      if constexpr (PHASE == 2) {
        if (a.base) {
          const Q4<float>* q = qb;
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            o[4 * mm] += a.gr * q[mm].x - a.gi * q[mm].y;
            o[4 * mm + 1] += a.gr * q[mm].y + a.gi * q[mm].x;
            o[4 * mm + 2] += a.gr * q[mm].z - a.gi * q[mm].w;
            o[4 * mm + 3] += a.gr * q[mm].w + a.gi * q[mm].z;
          }
        }
        if (a.prev) {
          Q4<float> q[4];
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) q[mm] = ld_chain_q4(a.prev + gz(g0 + T * mm));
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            o[4 * mm] += a.beta_prev * q[mm].x;
            o[4 * mm + 1] += a.beta_prev * q[mm].y;
            o[4 * mm + 2] += a.beta_prev * q[mm].z;
            o[4 * mm + 3] += a.beta_prev * q[mm].w;
          }
        }
        if (a.u_store) {
          Q4<float> q[4];
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) q[mm] = ld_stream_q4(a.u_store + gz(g0 + T * mm));
#pragma unroll
          for (int mm = 0; mm < 4; ++mm) {
            const Q4<float> r =
                apply_u(q[mm], Q4<float>{o[4 * mm], o[4 * mm + 1], o[4 * mm + 2], o[4 * mm + 3]});
            o[4 * mm] = r.x;
            o[4 * mm + 1] = r.y;
            o[4 * mm + 2] = r.z;
            o[4 * mm + 3] = r.w;
          }
        }
      }
      if (rows_out) {
#pragma unroll
        for (int mm = 0; mm < 4; ++mm)
          a.out[gz(g0 + T * mm)] = {o[4 * mm], o[4 * mm + 1], o[4 * mm + 2], o[4 * mm + 3]};
      } else if constexpr (PAIR) {
        if (h == 0) {
          tmem_st16(tres + (uint32_t)(16 * g), o);
        } else {
          float pa[16];
          tmem_ld16(tres + (uint32_t)(16 * g), pa);
          tmem_wait_ld_regs(pa);
          Q4<float>* dst = a.out + dst0 + 4 * g * dstep;
#pragma unroll
          for (int mm = 0; mm < 4; ++mm)
            if (dbg_in(dst0 + (4 * g + mm) * dstep + 1, (size_t)a.n_lines * L))
              st_points2(dst + mm * dstep, pa + 4 * mm, o + 4 * mm);
        }
      } else {
#pragma unroll
        for (int mm = 0; mm < 4; ++mm)
          reinterpret_cast<Q4<float>*>(tsm)[sz(lt * G::SPITCH + j + T * (4 * g + mm))] = {
              o[4 * mm], o[4 * mm + 1], o[4 * mm + 2], o[4 * mm + 3]};
      }
    }
    if constexpr (PAIR) {
      if (h == 0) {
        tmem_wait_st();
        h = 1;
      } else {
        h = 0;
        unit = next;
      }
    } else {
      __syncthreads();
      if (!rows_out) {
        const Q4<float>* st = reinterpret_cast<const Q4<float>*>(tsm);
        const int g = tid % LPC, i0 = tid / LPC;
        Q4<float>* dst = a.out + (size_t)i0 * a.n_lines + (unit * G::LPU + g);
        constexpr int RPI = G::THREADS / LPC;
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (dbg_in((size_t)(i0 + q * RPI) * a.n_lines + unit * G::LPU + g, (size_t)a.n_lines * L))
            dst[(size_t)(q * RPI) * a.n_lines] = st[sz(g * G::SPITCH + i0 + q * RPI)];
        __syncthreads();
      }
      unit = next;
      if (leader && unit < n_units) issue(unit, 0);
    }
  }
  if (failed && leader) {
    atomicExch(a.err, kErrTimeout);
    mbar_wait_bounded(bar, par ^ 1u, kWaitNs);  // the copy in flight
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (PAIR && warp == 0) tmem_dealloc(tbase, G::TCOLS);
}

}  // namespace dgb
