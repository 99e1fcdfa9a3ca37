// C ABI of the Scheme II library: context management and the host side of each call.
// Every numerical step runs in the kernels of this library; the host only validates,
// allocates, enqueues and copies.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <complex>
#include <cstring>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "../../include/dirac.h"
#include "ctx.h"
#include "internal.h"

using namespace dgb;



static thread_local std::string g_create_error;

namespace dgb {
void set_global_error(const std::string& msg) { g_create_error = msg; }
}  // namespace dgb

static size_t npts(const dirac_ctx* c) { return (size_t)c->nx * c->ny; }

static dirac_status fail(dirac_ctx* c, dirac_status s, const std::string& msg) {
  if (c) c->err = msg;
  else g_create_error = msg;
  return s;
}

static dirac_status cuda_fail(dirac_ctx* c, cudaError_t e, const char* where) {
  std::string m = std::string(where) + ": " + cudaGetErrorString(e);
  return fail(c, e == cudaErrorMemoryAllocation ? DIRAC_ENOMEM : DIRAC_ECUDA, m);
}

#define CK(call, where)                                   \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return cuda_fail(ctx, e_, where); \
  } while (0)

static bool pow2_in(int n, int lo, int hi) { return n >= lo && n <= hi && (n & (n - 1)) == 0; }

// Failure-detection test hook read at creation: DIRAC_FAULT=alloc:N (N >= 1) makes the
// N-th device allocation of the new context fail with cudaErrorMemoryAllocation, so the
// creation returns DIRAC_ENOMEM after freeing what it had allocated. Anything else: off.
static int fault_alloc_from_env() {
  const char* f = getenv("DIRAC_FAULT");
  if (!f || strncmp(f, "alloc:", 6) != 0) return 0;
  char* end = nullptr;
  const long n = strtol(f + 6, &end, 10);
  return (end && *end == '\0' && n >= 1 && n < (1L << 30)) ? (int)n : 0;
}

static cudaError_t dalloc(dirac_ctx* ctx, void** p, size_t bytes) {
  if (ctx->fault_alloc_at > 0 && ++ctx->n_allocs == ctx->fault_alloc_at) {
    // injected failure: nothing is allocated, the caller unwinds as for a real one
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaSuccess) ctx->allocs.push_back(*p);
  return e;
}

static void free_all(dirac_ctx* ctx) {
  if (ctx->k_host) cudaFreeHost(ctx->k_host);
  ctx->k_host = nullptr;
  for (void* p : ctx->allocs) cudaFree(p);
  ctx->allocs.clear();
}

// ------------------------------------------------------------------ precision dispatch
// launch option for a pass from the dirac_set_launch preference (0 = default)
static int pass_opt(const dirac_ctx* ctx, int shape, int L, int n_lines) {
  if (shape & DIRAC_LAUNCH_ALT_RADIX) {  // validated by dirac_set_launch
    const int threads = shape & ~DIRAC_LAUNCH_ALT_RADIX;
    if (ctx->prec == DIRAC_C64 ? line_pass_radix_alt<float>(L) : line_pass_radix_alt<double>(L))
      return threads == 256 ? 3 : 4;
    shape = threads;  // this line length has no alternative radix: the default one
  }
  const int threads = shape;
  if (threads == 256) return 0;
  if (threads == 512) return 1;
  if (threads == 1024) return 2;
  // Default, by measurement: complex64 the team pass for lines of 256 points or more (256^2
  // 0.0109 against 0.0118 ms per step for the radix-8 pass, 1024^2 0.0282 against 0.039); the
  // smaller shape for lines of 128 points or fewer, but for complex64 lines of 32 points or more
  // only below 2^17 points (smaller | larger x pass, ms per step: 32 x 2048 0.0135 | 0.0151, 64 x
  // 1024 0.0121 | 0.0118, 128 x 512 0.0127 | 0.0125, at 2^17 32 x 4096 0.0218 | 0.0200, 64 x 2048
  // 0.0170 | 0.0134, 128 x 1024 0.0137 | 0.0138, above it 128 x 2048 0.0202 | 0.0154), and, in
  // complex128, for 1024-point lines (one line per CTA: 1024 CTAs spread over the SMs to within
  // one line, 0.636 against 0.761 ms per 1024^2 step) and fewer than 512 lines of 512 points (512
  // x 256: 0.125 against 0.144 ms per step with both passes in one shape); else the larger.
  if (ctx->prec == DIRAC_C64) {
    if (L >= 256) return 2;
    return L >= 32 && (size_t)L * n_lines >= kWideShortLines ? 1 : 0;
  }
  return (L == 1024 || L <= 128 || (L == 512 && n_lines < 512)) ? 0 : 1;
}

// Reads and clears the device error flag (after the stream has been synchronised).
static dirac_status device_error(dirac_ctx* ctx) {
  int flag = 0;
  cudaError_t e = cudaMemcpy(&flag, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "read device error flag");
  if (DIRAC_DEBUG && dgb_debug_bounds())
    return fail(ctx, DIRAC_ECUDA, "debug build: an index check of a line pass failed");
  if (flag) {
    cudaMemset(ctx->d_err, 0, sizeof(int));
    return fail(ctx, DIRAC_ETIMEOUT, "a bounded device wait ran out; the state is not valid");
  }
  return DIRAC_OK;
}

template <typename T>
static LinePassArgs<T> pass_args(dirac_ctx* ctx, int axis) {
  LinePassArgs<T> a{};
  a.err = ctx->d_err;
  a.L = axis == 0 ? ctx->nx : ctx->ny;
  a.n_lines = axis == 0 ? ctx->ny : ctx->nx;
  a.sigma = axis;
  a.tw = (const Cx<T>*)(axis == 0 ? ctx->tw_x : ctx->tw_y);
  a.tw_alt = (const Cx<T>*)(axis == 0 ? ctx->tw_x_alt : ctx->tw_y_alt);
  a.tw_small = (const Cx<T>*)(axis == 0 ? ctx->tw_x_small : ctx->tw_y_small);
  a.tw_team = (const Cx<T>*)(axis == 0 ? ctx->tw_x_team : ctx->tw_y_team);
  return a;
}

// Scheme II with static potentials: whether the y pass' store applies the half steps that follow
// it (a team pass). The matrices are then kept in the transposed layout only; the launch shape
// decides it, so a step remakes them when dirac_set_launch or the autotuner changed that.
static bool pot_in_y_pass(const dirac_ctx* ctx) {
  return ctx->has_pot && ctx->scheme == DIRAC_SCHEME_II && ctx->prec == DIRAC_C64 &&
         team_length(ctx->ny) && pass_opt(ctx, ctx->threads_y, ctx->ny, ctx->nx) == 2;
}

template <typename T>
static dirac_status tables_for_dt(dirac_ctx* ctx, double dt) {
  cudaStream_t st = ctx->stream;
  ctx->dt_cached = 0.0;  // until they are complete
  const bool sym = ctx->scheme == DIRAC_SCHEME_II_SYMMETRIC;
  const bool need_u2n = ctx->scheme != DIRAC_SCHEME_II;  // U^2 applied in the normal layout
  if (sym && !ctx->mult_xh)
    CK(dalloc(ctx, &ctx->mult_xh, ctx->nx * sizeof(Q4<T>)), "allocate tables");
  if (sym && ctx->mult_px && !ctx->mult_pxh)
    CK(dalloc(ctx, &ctx->mult_pxh, ctx->nx * sizeof(Q4<T>)), "allocate tables");
  if (need_u2n && !ctx->u_identity && !ctx->u2_n)
    CK(dalloc(ctx, &ctx->u2_n, npts(ctx) * sizeof(Q4<T>)), "allocate half-step");
  if (!ctx->u_identity) {
    CK(launch_halfstep<T>(ctx->a1, ctx->a2, ctx->meff, ctx->omx, ctx->omy, ctx->nx, ctx->ny, dt,
                          (Q4<T>*)ctx->u_n, (Q4<T>*)ctx->u_t, (Q4<T>*)ctx->u2_t,
                          need_u2n ? (Q4<T>*)ctx->u2_n : nullptr, st),
       "half-step matrices");
    ctx->launches += 1;
  }
  if (ctx->has_pot) {
    if (!ctx->ug) CK(dalloc(ctx, &ctx->ug, 2 * npts(ctx) * sizeof(Q4<T>)), "allocate half-step");
    if (!ctx->ug2) CK(dalloc(ctx, &ctx->ug2, 2 * npts(ctx) * sizeof(Q4<T>)), "allocate half-step");
    ctx->ug_transposed = pot_in_y_pass(ctx);
    CK(launch_halfstep_general<T>(ctx->a1, ctx->a2, ctx->meff, ctx->omx, ctx->omy,
                                  ctx->pot_use[0] ? ctx->pot_v : nullptr,
                                  ctx->pot_use[1] ? ctx->pot_ax : nullptr,
                                  ctx->pot_use[2] ? ctx->pot_ay : nullptr, ctx->nx, ctx->ny, dt,
                                  ctx->ug_transposed, (Q4<T>*)ctx->ug, (Q4<T>*)ctx->ug2, st),
       "half-step matrices with potentials");
    ctx->launches += 1;
  }
  CK(launch_step_mult<T>(ctx->nx, ctx->ax, dt, (Q4<T>*)ctx->mult_x, st), "x multipliers");
  CK(launch_step_mult<T>(ctx->ny, ctx->ay, dt, (Q4<T>*)ctx->mult_y, st), "y multipliers");
  ctx->launches += 2;
  if (sym) {
    CK(launch_step_mult<T>(ctx->nx, ctx->ax, 0.5 * dt, (Q4<T>*)ctx->mult_xh, st),
       "x multipliers (dt/2)");
    ctx->launches += 1;
  }
  // the same tables in the team pass's order
  const void* perm_src[3] = {ctx->mult_x, ctx->mult_y, ctx->mult_xh};
  void* perm_dst[3] = {ctx->mult_px, ctx->mult_py, ctx->mult_pxh};
  for (int t = 0; t < 3; ++t) {
    if (!perm_dst[t]) continue;
    CK(launch_team_perm<T>(t == 1 ? ctx->ny : ctx->nx, (const Q4<T>*)perm_src[t],
                           (Q4<T>*)perm_dst[t], st),
       "multiplier order");
    ctx->launches += 1;
  }
  ctx->dt_cached = dt;
  return DIRAC_OK;
}

// psi <- U psi (squared = false) or U^2 psi in the normal layout, outside the passes: the
// general matrices when potentials are set, else the real-form ones (none when U = I).
template <typename T>
static dirac_status apply_half(dirac_ctx* ctx, void* psi, bool squared) {
  const size_t np = npts(ctx);
  if (ctx->has_pot) {
    const Q4<T>* ug = (const Q4<T>*)(squared ? ctx->ug2 : ctx->ug);
    if (ctx->ug_transposed)
      CK(launch_apply_ug_t<T>((Q4<T>*)psi, ug, ctx->nx, ctx->ny, ctx->stream), "half step");
    else
      CK(launch_apply_ug<T>((Q4<T>*)psi, ug, np, ctx->stream), "half step");
  } else if (!ctx->u_identity) {
    CK(launch_apply_u<T>((Q4<T>*)psi, (const Q4<T>*)(squared ? ctx->u2_n : ctx->u_n), np,
                         ctx->stream),
       "half step");
  } else {
    return DIRAC_OK;
  }
  ctx->launches += 1;
  return DIRAC_OK;
}

// Symmetric order: x over dt/2 (normal -> transposed), y over dt (transposed -> normal),
// x over dt/2 (normal -> normal, into the other buffer); U on the first x pass's load,
// U^2 / U on the last x pass's store. The state alternates between the two buffers and
// ends in ctx->psi.
template <typename T>
static dirac_status step_symmetric(dirac_ctx* ctx, long n) {
  LinePassArgs<T> ax = pass_args<T>(ctx, 0), ay = pass_args<T>(ctx, 1);
  ax.mult = (const Q4<T>*)ctx->mult_xh;
  ax.mult_perm = (const Q4<T>*)ctx->mult_pxh;
  ax.beta = (const T*)ctx->beta1;
  ax.beta_im = (const T*)ctx->beta1_im;
  ay.mult = (const Q4<T>*)ctx->mult_y;
  ay.mult_perm = (const Q4<T>*)ctx->mult_py;
  ay.beta = (const T*)ctx->beta2T;
  ay.beta_im = (const T*)ctx->beta2T_im;
  ax.test_extra_tx = ay.test_extra_tx = ctx->test_timeout_next;
  ctx->test_timeout_next = 0;
  void* cur = ctx->psi;
  void* oth = ctx->psiT;
  const int opt_x = pass_opt(ctx, ctx->threads_x, ctx->nx, ctx->ny);
  const int opt_y = pass_opt(ctx, ctx->threads_y, ctx->ny, ctx->nx);
  // potentials: as in step_impl, the later U in the last x pass's row store
  const bool fused = !ctx->has_pot;
  const bool fused_pot = !fused && sizeof(T) == 4 && opt_x == 2 && team_length(ctx->nx);
  if (!fused) {
    dirac_status r = apply_half<T>(ctx, cur, false);
    if (r != DIRAC_OK) return r;
  }
  for (long s = 0; s < n; ++s) {
    LinePassArgs<T> a1 = ax, a3 = ax;
    a1.in = (const Q4<T>*)cur;
    a1.out = (Q4<T>*)oth;
    a1.u_load = (fused && s == 0 && !ctx->u_identity) ? (const Q4<T>*)ctx->u_n : nullptr;
    ay.in = (const Q4<T>*)oth;
    ay.out = (Q4<T>*)cur;
    a3.in = (const Q4<T>*)cur;
    a3.out = (Q4<T>*)oth;
    a3.store_normal = 1;
    a3.u_store = (!fused || ctx->u_identity)
                     ? nullptr
                     : (const Q4<T>*)(s + 1 == n ? ctx->u_n : ctx->u2_n);
    a3.ug_store = fused_pot ? (const Q4<T>*)(s + 1 == n ? ctx->ug : ctx->ug2) : nullptr;
    CK(launch_line_pass<T>(a1, MODE_STEP, opt_x, ctx->stream), "x pass (dt/2)");
    CK(launch_line_pass<T>(ay, MODE_STEP, opt_y, ctx->stream), "y pass");
    CK(launch_line_pass<T>(a3, MODE_STEP, opt_x, ctx->stream), "x pass (dt/2, rows)");
    ctx->launches += 3;
    if (!fused && !fused_pot) {
      dirac_status r = apply_half<T>(ctx, oth, s + 1 < n);
      if (r != DIRAC_OK) return r;
    }
    void* t = cur;
    cur = oth;
    oth = t;
  }
  if (cur != ctx->psi) {  // the two state buffers trade names
    ctx->psiT = ctx->psi;
    ctx->psi = cur;
  }
  return DIRAC_OK;
}

// One application of the unsplit operator, S(v) = sum_j b^j sigma_j [[d_j]] v (so dt A = -dt S):
//   out = (ar + i ai) S(in) + (gr + i gi) base + beta prev, then U out if u is not null.
// `in` is in the normal (tr = false) or the transposed layout; out_rows: the result stays in
// the layout of the second pass' rows, the other one than `in`'s; otherwise it returns to the
// layout of `in`. base, prev and u are in the layout of the rows; in_t receives `in` in that
// layout (base may be in_t).
struct UnsplitOp {
  const void* in = nullptr;
  bool tr = false;
  void* in_t = nullptr;
  void* out = nullptr;
  bool out_rows = false;
  double ar = 0.0, ai = 0.0;
  const void* base = nullptr;
  double gr = 0.0, gi = 0.0;
  const void* prev = nullptr;
  double beta = 0.0;
  const void* u = nullptr;
};

// complex64 grids whose axes both have team-pass lengths run the operator as two team passes,
// with the result in either layout; the others as two derivative passes, a transpose and a
// pointwise combine, everything in the normal layout.
static bool unsplit_team(const dirac_ctx* ctx) {
  return ctx->prec == DIRAC_C64 && ctx->dmult_px && ctx->dmult_py && !ctx->beta1_im;
}

// in -> out through two team passes; scratch1 holds the first axis' term.
static dirac_status unsplit_apply_team(dirac_ctx* ctx, const UnsplitOp& op) {
  cudaStream_t st = ctx->stream;
  for (int phase = 1; phase <= 2; ++phase) {
    UnsplitArgs a{};
    a.axis = (phase == 1) == op.tr ? 1 : 0;  // phase 1 runs along the rows of `in`
    a.n_lines = a.axis == 0 ? ctx->ny : ctx->nx;
    a.beta = (const float*)(a.axis == 0 ? ctx->beta1 : ctx->beta2T);
    a.tw = (const Cx<float>*)(a.axis == 0 ? ctx->tw_x_team : ctx->tw_y_team);
    a.mult = (const Q4<float>*)(a.axis == 0 ? ctx->dmult_px : ctx->dmult_py);
    a.err = ctx->d_err;
    if (phase == 1) {
      a.in = (const Q4<float>*)op.in;
      a.out = (Q4<float>*)ctx->scratch1;
      a.out_in = (Q4<float>*)op.in_t;
      a.test_extra_tx = ctx->test_timeout_next;
      ctx->test_timeout_next = 0;
    } else {
      a.in = (const Q4<float>*)op.in_t;
      a.out = (Q4<float>*)op.out;
      a.s_other = (const Q4<float>*)ctx->scratch1;
      a.ar = (float)op.ar;
      a.ai = (float)op.ai;
      a.base = (const Q4<float>*)op.base;
      a.gr = (float)op.gr;
      a.gi = (float)op.gi;
      a.prev = (const Q4<float>*)op.prev;
      a.beta_prev = (float)op.beta;
      a.u_store = (const Q4<float>*)op.u;
      a.store_normal = op.out_rows ? 1 : 0;
    }
    CK(launch_unsplit(a, a.axis == 0 ? ctx->nx : ctx->ny, phase, st), "unsplit operator");
  }
  ctx->launches += 2;
  return DIRAC_OK;
}

// The general path: normal layout throughout (op.tr, op.in_t, op.out_rows and op.u unused, base
// and prev in the normal layout). psiT, scratch1 and scratch2 are scratch.
template <typename T>
static dirac_status unsplit_apply(dirac_ctx* ctx, const UnsplitOp& op) {
  cudaStream_t st = ctx->stream;
  ctx->test_timeout_next = 0;  // no bounded waits here
  LinePassArgs<T> ax = pass_args<T>(ctx, 0), ay = pass_args<T>(ctx, 1);
  ax.in = (const Q4<T>*)op.in;
  ax.out = (Q4<T>*)ctx->scratch1;
  ax.mult = (const Q4<T>*)ctx->dmult_x;
  ax.store_normal = 1;
  CK(launch_line_pass<T>(ax, MODE_DERIV, 0, st), "x derivative");
  CK(launch_transpose<T>((const Q4<T>*)op.in, (Q4<T>*)ctx->psiT, ctx->ny, ctx->nx, st),
     "transpose");
  ay.in = (const Q4<T>*)ctx->psiT;
  ay.out = (Q4<T>*)ctx->scratch2;
  ay.mult = (const Q4<T>*)ctx->dmult_y;
  CK(launch_line_pass<T>(ay, MODE_DERIV, 0, st), "y derivative");
  CK(launch_unsplit_combine<T>((const Q4<T>*)ctx->scratch1, (const Q4<T>*)ctx->scratch2, ctx->a1,
                               ctx->a2, ctx->sxinv, ctx->syinv, ctx->sxinv_im, ctx->syinv_im,
                               ctx->nx, ctx->ny, op.ar, op.ai, (const Q4<T>*)op.base, op.gr,
                               op.gi, (const Q4<T>*)op.prev, op.beta, (Q4<T>*)op.out, st),
     "combine");
  ctx->launches += 4;
  return DIRAC_OK;
}

#define CKS(x)                       \
  do {                               \
    dirac_status s_ = (x);           \
    if (s_ != DIRAC_OK) return s_;   \
  } while (0)

// The polynomial scheme (eq. poly): U, the middle step, U per step, with U^2 between
// consecutive steps of a call. The middle step's sum is evaluated from its highest term down,
// so that no separate sum is kept: Taylor by Horner's rule, t <- psi + (dt/q) A t for q = N..1;
// Chebyshev by Clenshaw's recurrence, b_k = c_k psi + 2 B b_{k+1} - b_{k+2}, the sum being
// c_0 psi + B b_1 - b_2, with B = (i dt / R) A = -(i dt / R) S, c_k = (2 - delta_k0) (-i)^k
// J_k(R) and b_N = c_N psi (folded into the factors of the first two applications). The team
// passes alternate the layout of the terms; b_{k+2} is then always in the layout of b_k.
template <typename T>
static dirac_status step_poly(dirac_ctx* ctx, long n, double dt) {
  cudaStream_t st = ctx->stream;
  const size_t np = npts(ctx), bytes = np * sizeof(Q4<T>);
  for (void*& p : ctx->pool)
    if (!p) CK(dalloc(ctx, &p, bytes), "allocate polynomial terms");
  if (!ctx->scratch1) CK(dalloc(ctx, &ctx->scratch1, bytes), "scratch");
  if (!ctx->scratch2) CK(dalloc(ctx, &ctx->scratch2, bytes), "scratch");
  const int N = ctx->poly_degree;
  const bool cheb = ctx->scheme == DIRAC_SCHEME_POLY_CHEBYSHEV;
  std::vector<double> jq(N + 1, 0.0);
  double R = 0.0;
  if (cheb) {
    if (ctx->bmax[0] < 0.0) {  // max |b^j| over the grid, once per context
      const int nb = 256;
      double* part = nullptr;
      CK(dalloc(ctx, (void**)&part, 2 * nb * sizeof(double)), "scratch");
      CK(launch_max_b(ctx->a1, ctx->a2, ctx->sxinv, ctx->syinv, ctx->sxinv_im, ctx->syinv_im,
                      ctx->nx, ctx->ny, part, nb, st),
         "max b");
      std::vector<double> h(2 * nb);
      CK(cudaMemcpyAsync(h.data(), part, 2 * nb * sizeof(double), cudaMemcpyDeviceToHost, st),
         "max b");
      CK(cudaStreamSynchronize(st), "max b");
      ctx->bmax[0] = ctx->bmax[1] = 0.0;
      for (int b = 0; b < nb; ++b) {
        ctx->bmax[0] = fmax(ctx->bmax[0], h[2 * b]);
        ctx->bmax[1] = fmax(ctx->bmax[1], h[2 * b + 1]);
      }
      ctx->launches += 1;
    }
    const double hx = 2.0 * ctx->ax / ctx->nx, hy = 2.0 * ctx->ay / ctx->ny;
    R = dt * (ctx->bmax[0] * M_PI / hx + ctx->bmax[1] * M_PI / hy);
    if (!(R > 0.0) || !bessel_j_series(R, N, jq.data()))
      return fail(ctx, DIRAC_EINVAL, "no Chebyshev bound for this grid and dt");
  }
  using cd = std::complex<double>;
  auto c_of = [&](int k) {  // (2 - delta_k0) (-i)^k J_k
    static const double pr[4] = {1.0, 0.0, -1.0, 0.0}, pi_[4] = {0.0, -1.0, 0.0, 1.0};
    return (k == 0 ? 1.0 : 2.0) * jq[k] * cd(pr[k & 3], pi_[k & 3]);
  };
  const bool team = unsplit_team(ctx);
  for (long s = 0; s < n; ++s) {
    if (s == 0) CKS(apply_half<T>(ctx, ctx->psi, false));
    const bool last_step = s + 1 == n;
    // U after the middle step, inside the last application where it can be
    const bool fuse_u = team && !ctx->has_pot && !ctx->u_identity;
    const void *cur = ctx->psi, *prev = nullptr;  // b_{k+1}, b_{k+2}
    for (int i = 1; i <= N; ++i) {  // application i makes term k = N - i
      const int k = N - i;
      UnsplitOp op;
      op.in = cur;
      op.tr = team && i % 2 == 0;
      cd al, ga;
      if (!cheb) {
        al = -dt / (k + 1);
        ga = 1.0;
      } else {
        al = cd(0.0, -dt / R) * (k == 0 ? 1.0 : 2.0);
        ga = c_of(k);
        if (i == 1) al *= c_of(N);
        if (i == 2) ga -= c_of(N);
        if (i >= 3) {
          op.prev = prev;
          op.beta = -1.0;
        }
      }
      op.ar = al.real();
      op.ai = al.imag();
      op.gr = ga.real();
      op.gi = ga.imag();
      int slot = 0;  // a buffer that holds neither b_{k+1} nor b_{k+2}
      while (ctx->pool[slot] == cur || ctx->pool[slot] == prev) ++slot;
      op.out = ctx->pool[slot];
      if (team) {
        const bool rows_tr = !op.tr;  // the second pass' rows are in the transposed layout
        op.in_t = i == 1 ? ctx->psiT : ctx->scratch2;
        op.base = rows_tr ? ctx->psiT : ctx->psi;
        op.out_rows = !(i == N && rows_tr);  // the sum ends in the normal layout
        if (i == N && fuse_u)
          op.u = rows_tr ? (last_step ? ctx->u_t : ctx->u2_t) : (last_step ? ctx->u_n : ctx->u2_n);
        CKS(unsplit_apply_team(ctx, op));
      } else {
        op.base = ctx->psi;
        CKS(unsplit_apply<T>(ctx, op));
      }
      prev = cur;
      cur = op.out;
      if (i == 1) prev = nullptr;  // b_N is never stored
    }
    // the sum is the new state; the old state's buffer joins the pool
    for (void*& p : ctx->pool)
      if (p == cur) {
        p = ctx->psi;
        break;
      }
    ctx->psi = (void*)cur;
    if (!fuse_u) CKS(apply_half<T>(ctx, ctx->psi, !last_step));
  }
  return DIRAC_OK;
}

// ---- Scheme I (eq. cn): U, G psi* = G~ psi by restarted GMRES, U (U^2 between steps).
// G v = v - dt/2 A v = v + dt/2 S(v), G~ v = v - dt/2 S(v) (S as in unsplit_apply).
constexpr int kKrylovBlocks = 608;

// out = v + a S(v), normal layout
template <typename T>
static dirac_status cn_apply(dirac_ctx* ctx, const void* v, void* out, double a) {
  UnsplitOp op;
  op.in = v;
  op.out = out;
  op.ar = a;
  op.gr = 1.0;
  op.in_t = ctx->psiT;
  if (unsplit_team(ctx)) {
    op.base = ctx->psiT;  // the transposed copy of v
    return unsplit_apply_team(ctx, op);
  }
  op.base = v;
  return unsplit_apply<T>(ctx, op);
}

// Waits until the dot products, which the normalisation writes, are in the pinned host buffer.
// DIRAC_ETIMEOUT if a bounded wait ran out in the operator's passes: what they left is not to
// be iterated on.
static dirac_status krylov_fetch(dirac_ctx* ctx) {
  CK(cudaStreamSynchronize(ctx->stream), "inner products");
  return ctx->k_host[kKrylovErr] != 0.0 ? device_error(ctx) : DIRAC_OK;
}

// out += sum_{i < c.size()} c_i V_i
template <typename T>
static dirac_status krylov_combine(dirac_ctx* ctx, void* out,
                                   const std::vector<std::complex<double>>& c) {
  double* h = ctx->k_host + kKrylovHost / 2;  // not read by the device at this point
  for (size_t i = 0; i < c.size(); ++i) {
    h[2 * i] = c[i].real();
    h[2 * i + 1] = c[i].imag();
  }
  CK(cudaMemcpyAsync(ctx->k_coef, h, 2 * c.size() * sizeof(double), cudaMemcpyHostToDevice,
                     ctx->stream),
     "coefficients");
  CK(launch_multi_axpy<T>((Q4<T>*)out, (const Q4<T>* const*)ctx->k_vptr, ctx->k_coef,
                          (int)c.size(), npts(ctx), ctx->stream),
     "combination");
  ctx->launches += 1;
  return DIRAC_OK;
}

// One Arnoldi step after w = G V_j is in kv[j + 1]: classical Gram-Schmidt twice against V_0..V_j
// and the norm, everything on the device. dots: h (2 m values), second h (2 m), norm^2, 1/norm.
// fp64: the sums of complex64 vectors in FP64.
template <typename T>
static dirac_status krylov_orthogonalise(dirac_ctx* ctx, int m, bool fp64) {
  cudaStream_t st = ctx->stream;
  const size_t np = npts(ctx);
  const auto V = (const Q4<T>* const*)ctx->k_vptr;
  Q4<T>* w = (Q4<T>*)ctx->kv[m];
  double *d0 = ctx->k_dots, *d1 = d0 + 2 * m, *d2 = d1 + 2 * m;
  CK(launch_gram_schmidt<T>(0, fp64, V, m, w, nullptr, np, ctx->k_partials, ctx->k_ticket, d0,
                            kKrylovBlocks, st),
     "inner products");
  if (m <= 4) {
    // the first combination and the second products in one sweep
    CK(launch_gram_schmidt<T>(1, fp64, V, m, w, d0, np, ctx->k_partials, ctx->k_ticket, d1,
                              kKrylovBlocks, st),
       "inner products");
  } else {
    CK(launch_gram_schmidt<T>(2, fp64, V, m, w, d0, np, ctx->k_partials, ctx->k_ticket, d2,
                              kKrylovBlocks, st),
       "combination");
    CK(launch_gram_schmidt<T>(0, fp64, V, m, w, nullptr, np, ctx->k_partials, ctx->k_ticket, d1,
                              kKrylovBlocks, st),
       "inner products");
    ctx->launches += 1;
  }
  CK(launch_gram_schmidt<T>(2, fp64, V, m, w, d1, np, ctx->k_partials, ctx->k_ticket, d2, kKrylovBlocks,
                            st),
     "combination");
  CK(launch_normalise<T>(w, d0, 4 * m + 1, ctx->d_err, ctx->k_host, ctx->k_host + kKrylovErr, np,
                         st), "normalise");
  ctx->launches += 4;
  return DIRAC_OK;
}

template <typename T>
static dirac_status step_cn(dirac_ctx* ctx, long n, double dt) {
  cudaStream_t st = ctx->stream;
  const size_t np = npts(ctx), bytes = np * sizeof(Q4<T>);
  const int m = ctx->krylov_m;
  const double tol = ctx->krylov_tol > 0.0 ? ctx->krylov_tol : (sizeof(T) == 8 ? 1e-14 : 3e-7);
  // buffers: basis V_0..V_m, the right-hand side, the pointer table of the basis
  while ((int)ctx->kv.size() < m + 1) {
    void* p = nullptr;
    CK(dalloc(ctx, &p, bytes), "allocate Krylov basis");
    ctx->kv.push_back(p);
  }
  if (!ctx->k_rhs) CK(dalloc(ctx, &ctx->k_rhs, bytes), "allocate Krylov basis");
  if (!ctx->scratch1) CK(dalloc(ctx, &ctx->scratch1, bytes), "scratch");
  if (!ctx->scratch2) CK(dalloc(ctx, &ctx->scratch2, bytes), "scratch");
  if (!ctx->k_partials)
    CK(dalloc(ctx, (void**)&ctx->k_partials, 2 * (size_t)kKrylovBlocks * 102 * sizeof(double)),
       "scratch");
  if (!ctx->k_coef) CK(dalloc(ctx, (void**)&ctx->k_coef, 2 * 102 * sizeof(double)), "scratch");
  if (!ctx->k_dots) CK(dalloc(ctx, (void**)&ctx->k_dots, kKrylovHost * sizeof(double)), "scratch");
  if (!ctx->k_vptr) CK(dalloc(ctx, (void**)&ctx->k_vptr, 102 * sizeof(void*)), "scratch");
  if (!ctx->k_host)
    CK(cudaMallocHost((void**)&ctx->k_host, kKrylovHost * sizeof(double)), "scratch");
  if (!ctx->k_ticket) {
    CK(dalloc(ctx, (void**)&ctx->k_ticket, sizeof(unsigned)), "scratch");
    CK(cudaMemsetAsync(ctx->k_ticket, 0, sizeof(unsigned), st), "scratch");
  }
  CK(cudaMemcpyAsync(ctx->k_vptr, ctx->kv.data(), (m + 1) * sizeof(void*), cudaMemcpyHostToDevice,
                     st),
     "pointer table");
  using cd = std::complex<double>;
  std::vector<cd> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
  for (long s = 0; s < n; ++s) {
    if (s == 0) CKS(apply_half<T>(ctx, ctx->psi, false));
    void* x = ctx->psi;
    CKS(cn_apply<T>(ctx, x, ctx->k_rhs, -0.5 * dt));
    double bnorm = 0.0;
    bool converged = false;
    for (int cycle = 0; cycle <= ctx->krylov_restarts && !converged; ++cycle) {
      // r = rhs - G x into V_0; for the initial guess psi, G~ psi - G psi = 2 (rhs - psi)
      void* v0 = ctx->kv[0];
      if (cycle > 0) CKS(cn_apply<T>(ctx, x, v0, 0.5 * dt));
      CK(launch_residual<T>(cycle > 0 ? 1 : 0, (const Q4<T>*)ctx->k_rhs, (const Q4<T>*)x,
                            (Q4<T>*)v0, np, ctx->k_partials, ctx->k_ticket, ctx->k_dots,
                            kKrylovBlocks, st),
         "residual");
      CK(launch_normalise<T>((Q4<T>*)v0, ctx->k_dots, 2, ctx->d_err, ctx->k_host,
                             ctx->k_host + kKrylovErr, np, st), "normalise");
      ctx->launches += 2;
      CKS(krylov_fetch(ctx));
      const double beta = sqrt(fmax(ctx->k_host[0], 0.0));
      if (cycle == 0) bnorm = sqrt(ctx->k_host[1]);
      if (beta <= tol * bnorm || beta == 0.0) {
        converged = true;
        break;
      }
      if (cycle == ctx->krylov_restarts) break;
      std::fill(g.begin(), g.end(), cd(0.0));
      g[0] = beta;
      int kdim = 0;
      for (int j = 0; j < m; ++j) {
        // FP32 sums hold |w| up to about 1e19; a larger one (a time step of that many periods of
        // the fastest mode) overflows them, and the vector is made again with FP64 sums
        for (bool fp64 : {false, true}) {
          CKS(cn_apply<T>(ctx, ctx->kv[j], ctx->kv[j + 1], 0.5 * dt));
          CKS(krylov_orthogonalise<T>(ctx, j + 1, fp64));
          CKS(krylov_fetch(ctx));
          if (sizeof(T) == 8 || std::all_of(ctx->k_host, ctx->k_host + 4 * (j + 1) + 1,
                                            [](double v) { return isfinite(v); }))
            break;
        }
        const double* d = ctx->k_host;
        for (int i = 0; i <= j; ++i)
          H[(size_t)i * m + j] = cd(d[2 * i], d[2 * i + 1]) +
                                 cd(d[2 * (j + 1) + 2 * i], d[2 * (j + 1) + 2 * i + 1]);
        const double hn = sqrt(fmax(d[4 * (j + 1)], 0.0));
        H[(size_t)(j + 1) * m + j] = hn;
        for (int i = 0; i < j; ++i) {  // earlier Givens rotations on column j
          const cd a = H[(size_t)i * m + j], b = H[(size_t)(i + 1) * m + j];
          H[(size_t)i * m + j] = std::conj(cs[i]) * a + std::conj(sn[i]) * b;
          H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * b;
        }
        const cd a = H[(size_t)j * m + j], b = H[(size_t)(j + 1) * m + j];
        const double r = sqrt(std::norm(a) + std::norm(b));
        cs[j] = r > 0.0 ? a / r : cd(1.0);
        sn[j] = r > 0.0 ? b / r : cd(0.0);
        H[(size_t)j * m + j] = r;
        H[(size_t)(j + 1) * m + j] = 0.0;
        g[j + 1] = -sn[j] * g[j];
        g[j] = std::conj(cs[j]) * g[j];
        kdim = j + 1;
        ctx->krylov_iters += 1;
        if (std::abs(g[j + 1]) <= tol * bnorm || hn == 0.0) break;
      }
      for (int i = kdim - 1; i >= 0; --i) {  // H y = g, then x += V y
        cd acc = g[i];
        for (int t = i + 1; t < kdim; ++t) acc -= H[(size_t)i * m + t] * y[t];
        y[i] = acc / H[(size_t)i * m + i];
      }
      CKS(krylov_combine<T>(ctx, x, std::vector<cd>(y.begin(), y.begin() + kdim)));
    }
    if (!converged) return fail(ctx, DIRAC_ENOCONV, "Scheme I: GMRES did not converge");
    CKS(apply_half<T>(ctx, ctx->psi, s + 1 < n));
  }
  return DIRAC_OK;
}

// Contexts whose Scheme II steps run whole inside one launch (small_steps.cu): default launch
// shapes, no static potentials.
static bool whole_steps(const dirac_ctx* ctx, bool any_shape = false) {
  return ctx->prec == DIRAC_C64 && ctx->scheme == DIRAC_SCHEME_II && !ctx->has_pot &&
         !ctx->beta1_im && (any_shape || (!ctx->threads_x && !ctx->threads_y)) &&
         small_steps_grid(ctx->nx, ctx->ny);
}

// n steps in launches of at most kSmallSteps (a few milliseconds each); *done = false if the
// device cannot hold the cluster (the steps then run as separate passes).
constexpr long kSmallSteps = 1024;
static dirac_status step_small(dirac_ctx* ctx, long n, bool* done) {
  SmallStepArgs a{};
  a.psi = (Q4<float>*)ctx->psi;
  a.beta1 = (const float*)ctx->beta1;
  a.beta2 = (const float*)ctx->beta2T;
  a.u_n = ctx->u_identity ? nullptr : (const Q4<float>*)ctx->u_n;
  a.u_t = ctx->u_identity ? nullptr : (const Q4<float>*)ctx->u_t;
  a.u2_t = ctx->u_identity ? nullptr : (const Q4<float>*)ctx->u2_t;
  a.mult_x = (const Q4<float>*)ctx->mult_x;
  a.mult_y = (const Q4<float>*)ctx->mult_y;
  a.tw_x = (const Cx<float>*)ctx->tw_x;
  a.tw_y = (const Cx<float>*)ctx->tw_y;
  *done = false;
  for (long s = 0; s < n; s += kSmallSteps) {
    const long k = n - s < kSmallSteps ? n - s : kSmallSteps;
    const cudaError_t e = launch_small_steps(a, ctx->nx, ctx->ny, (int)k, s == 0, s + k == n,
                                             ctx->stream);
    if (e == cudaErrorNotSupported && s == 0) return DIRAC_OK;
    CK(e, "steps");
    ctx->launches += 1;
  }
  ctx->test_timeout_next = 0;
  *done = true;
  return DIRAC_OK;
}

template <typename T>
static dirac_status step_impl(dirac_ctx* ctx, long n, double dt) {
  if (dt != ctx->dt_cached || (ctx->has_pot && ctx->ug_transposed != pot_in_y_pass(ctx))) {
    dirac_status s = tables_for_dt<T>(ctx, dt);
    if (s != DIRAC_OK) return s;
  }
  if (ctx->scheme == DIRAC_SCHEME_II_SYMMETRIC) return step_symmetric<T>(ctx, n);
  if (ctx->scheme == DIRAC_SCHEME_POLY_TAYLOR || ctx->scheme == DIRAC_SCHEME_POLY_CHEBYSHEV)
    return step_poly<T>(ctx, n, dt);
  if (ctx->scheme == DIRAC_SCHEME_CRANK_NICOLSON) return step_cn<T>(ctx, n, dt);
  if (sizeof(T) == 4 && whole_steps(ctx)) {
    bool done = false;
    CKS(step_small(ctx, n, &done));
    if (done) return DIRAC_OK;
  }
  LinePassArgs<T> ax = pass_args<T>(ctx, 0), ay = pass_args<T>(ctx, 1);
  ax.in = (const Q4<T>*)ctx->psi;
  ax.out = (Q4<T>*)ctx->psiT;
  ax.mult = (const Q4<T>*)ctx->mult_x;
  ax.mult_perm = (const Q4<T>*)ctx->mult_px;
  ax.beta = (const T*)ctx->beta1;
  ax.beta_im = (const T*)ctx->beta1_im;
  ay.in = (const Q4<T>*)ctx->psiT;
  ay.out = (Q4<T>*)ctx->psi;
  ay.mult = (const Q4<T>*)ctx->mult_y;
  ay.mult_perm = (const Q4<T>*)ctx->mult_py;
  ay.beta = (const T*)ctx->beta2T;
  ay.beta_im = (const T*)ctx->beta2T_im;
  ax.test_extra_tx = ay.test_extra_tx = ctx->test_timeout_next;
  ctx->test_timeout_next = 0;
  // potentials: the leading U by its own kernel, the later ones in the y pass's store where
  // that is a team pass, else by their own kernel too
  const bool fused = !ctx->has_pot;
  const int opt_y = pass_opt(ctx, ctx->threads_y, ctx->ny, ctx->nx);
  const bool fused_pot = !fused && ctx->ug_transposed;
  if (!fused) CKS(apply_half<T>(ctx, ctx->psi, false));
  for (long s = 0; s < n; ++s) {
    ax.u_load = (fused && s == 0 && !ctx->u_identity) ? (const Q4<T>*)ctx->u_n : nullptr;
    ax.u_store = nullptr;
    CK(launch_line_pass<T>(ax, MODE_STEP, pass_opt(ctx, ctx->threads_x, ctx->nx, ctx->ny), ctx->stream),
       "x pass");
    ay.u_load = nullptr;
    ay.u_store = (!fused || ctx->u_identity) ? nullptr
                                             : (const Q4<T>*)(s + 1 == n ? ctx->u_t : ctx->u2_t);
    ay.ug_store = fused_pot ? (const Q4<T>*)(s + 1 == n ? ctx->ug : ctx->ug2) : nullptr;
    CK(launch_line_pass<T>(ay, MODE_STEP, opt_y, ctx->stream), "y pass");
    ctx->launches += 2;
    if (!fused && !fused_pot) CKS(apply_half<T>(ctx, ctx->psi, s + 1 < n));
  }
  return DIRAC_OK;
}

// Spectral derivatives of the state: dx (normal layout) into scratch1, dy into scratch2.
template <typename T>
static dirac_status state_derivatives(dirac_ctx* ctx) {
  cudaStream_t st = ctx->stream;
  LinePassArgs<T> ax = pass_args<T>(ctx, 0), ay = pass_args<T>(ctx, 1);
  // y derivative: transpose psi -> scratch1 ([nx][ny]); derivative pass stores it back
  // transposed, i.e. in the normal layout, into scratch2.
  CK(launch_transpose<T>((const Q4<T>*)ctx->psi, (Q4<T>*)ctx->scratch1, ctx->ny, ctx->nx, st),
     "transpose");
  ay.in = (const Q4<T>*)ctx->scratch1;
  ay.out = (Q4<T>*)ctx->scratch2;
  ay.mult = (const Q4<T>*)ctx->dmult_y;
  CK(launch_line_pass<T>(ay, MODE_DERIV, 0, st), "y derivative");
  // x derivative: rows in the normal layout into scratch1.
  ax.in = (const Q4<T>*)ctx->psi;
  ax.out = (Q4<T>*)ctx->scratch1;
  ax.mult = (const Q4<T>*)ctx->dmult_x;
  ax.store_normal = 1;
  CK(launch_line_pass<T>(ax, MODE_DERIV, 0, st), "x derivative");
  ctx->launches += 3;
  return DIRAC_OK;
}

template <typename T>
static dirac_status observables_impl(dirac_ctx* ctx, dirac_obs* out, double* density_host) {
  cudaStream_t st = ctx->stream;
  const size_t n = npts(ctx);
  if (!ctx->scratch1) {
    CK(dalloc(ctx, &ctx->scratch1, n * sizeof(Q4<T>)), "scratch");
    CK(dalloc(ctx, &ctx->scratch2, n * sizeof(Q4<T>)), "scratch");
  }
  dirac_status s = state_derivatives<T>(ctx);
  if (s != DIRAC_OK) return s;
  if (density_host && !ctx->density) CK(dalloc(ctx, (void**)&ctx->density, n * sizeof(double)), "density");
  const int blocks = observables_blocks(n);
  CK(launch_observables<T>((const Q4<T>*)ctx->psi, (const Q4<T>*)ctx->scratch1,
                           (const Q4<T>*)ctx->scratch2, ctx->a1, ctx->a2, ctx->meff, ctx->w,
                           ctx->omx, ctx->omy, ctx->pot_use[0] ? ctx->pot_v : nullptr,
                           ctx->pot_use[1] ? ctx->pot_ax : nullptr,
                           ctx->pot_use[2] ? ctx->pot_ay : nullptr, n,
                           density_host ? ctx->density : nullptr, ctx->partials, blocks, st),
     "observables");
  const double hxhy = (2.0 * ctx->ax / ctx->nx) * (2.0 * ctx->ay / ctx->ny);
  CK(launch_reduce_partials(ctx->partials, blocks, hxhy, ctx->result, st), "reduce");
  ctx->launches += 2;
  double r[4];
  CK(cudaMemcpyAsync(r, ctx->result, sizeof(r), cudaMemcpyDeviceToHost, st), "copy result");
  if (density_host)
    CK(cudaMemcpyAsync(density_host, ctx->density, n * sizeof(double), cudaMemcpyDeviceToHost, st),
       "copy density");
  CK(cudaStreamSynchronize(st), "synchronize");
  {
    dirac_status de = device_error(ctx);
    if (de != DIRAC_OK) return de;
  }
  out->norm = r[0];
  out->norm_gamma = r[1];
  out->energy = r[2];
  out->energy_imag = r[3];
  if (!isfinite(r[0]) || !isfinite(r[1]) || !isfinite(r[2]) || !isfinite(r[3]))
    return fail(ctx, DIRAC_ENONFINITE, "the state holds non-finite values");
  return DIRAC_OK;
}

template <typename T>
static dirac_status create_impl(dirac_ctx* ctx, const double* g_host[3]) {
  cudaStream_t st = ctx->stream;
  const size_t n = npts(ctx);
  const int nx = ctx->nx, ny = ctx->ny;
  // FP64 fields
  double** f64[] = {&ctx->a1, &ctx->a2, &ctx->meff, &ctx->w, &ctx->omx, &ctx->omy};
  for (double** p : f64) CK(dalloc(ctx, (void**)p, n * sizeof(double)), "allocate fields");
  const bool complex_layer =
      ctx->abs.theta != 0.0 && (ctx->abs.width_x > 0 || ctx->abs.width_y > 0);
  // state, coefficient fields, tables
  CK(dalloc(ctx, &ctx->psi, n * sizeof(Q4<T>)), "allocate state");
  CK(dalloc(ctx, &ctx->psiT, n * sizeof(Q4<T>)), "allocate state");
  CK(dalloc(ctx, &ctx->beta1, n * sizeof(T)), "allocate coefficients");
  CK(dalloc(ctx, &ctx->beta2T, n * sizeof(T)), "allocate coefficients");
  if (complex_layer) {
    CK(dalloc(ctx, &ctx->beta1_im, n * sizeof(T)), "allocate coefficients");
    CK(dalloc(ctx, &ctx->beta2T_im, n * sizeof(T)), "allocate coefficients");
  }
  if (!ctx->u_identity) {
    CK(dalloc(ctx, &ctx->u_n, n * sizeof(Q4<T>)), "allocate half-step");
    CK(dalloc(ctx, &ctx->u_t, n * sizeof(Q4<T>)), "allocate half-step");
    CK(dalloc(ctx, &ctx->u2_t, n * sizeof(Q4<T>)), "allocate half-step");
  }
  // the per-axis tables and small buffers share one allocation (each cudaMalloc costs as much as
  // several of the kernels that fill them)
  std::vector<std::pair<void**, size_t>> small;
  auto table = [&](void* p, size_t bytes) { small.push_back({(void**)p, bytes}); };
  table(&ctx->sxinv, nx * sizeof(double));
  table(&ctx->syinv, ny * sizeof(double));
  if (complex_layer) {
    table(&ctx->sxinv_im, nx * sizeof(double));
    table(&ctx->syinv_im, ny * sizeof(double));
  }
  table(&ctx->tw_x, nx * sizeof(Cx<T>));
  table(&ctx->tw_y, ny * sizeof(Cx<T>));
  if (line_pass_radix_alt<T>(nx)) table(&ctx->tw_x_alt, nx * sizeof(Cx<T>));
  if (line_pass_radix_alt<T>(ny)) table(&ctx->tw_y_alt, ny * sizeof(Cx<T>));
  if (line_pass_radix_small<T>(nx, ny)) table(&ctx->tw_x_small, nx * sizeof(Cx<T>));
  if (line_pass_radix_small<T>(ny, nx)) table(&ctx->tw_y_small, ny * sizeof(Cx<T>));
  table(&ctx->mult_x, nx * sizeof(Q4<T>));
  table(&ctx->mult_y, ny * sizeof(Q4<T>));
  table(&ctx->dmult_x, nx * sizeof(Q4<T>));
  table(&ctx->dmult_y, ny * sizeof(Q4<T>));
  if (sizeof(T) == 4 && team_length(nx)) {  // the team pass's table orders and twiddles
    table(&ctx->mult_px, nx * sizeof(Q4<T>));
    table(&ctx->dmult_px, nx * sizeof(Q4<T>));
    table(&ctx->tw_x_team, nx * sizeof(Cx<T>));
  }
  if (sizeof(T) == 4 && team_length(ny)) {
    table(&ctx->mult_py, ny * sizeof(Q4<T>));
    table(&ctx->dmult_py, ny * sizeof(Q4<T>));
    table(&ctx->tw_y_team, ny * sizeof(Cx<T>));
  }
  table(&ctx->partials, 4 * sizeof(double) * observables_blocks(n));
  table(&ctx->result, 4 * sizeof(double));
  table(&ctx->d_err, sizeof(int));
  size_t total = 0;
  for (auto& t : small) total += (t.second + 255) / 256 * 256;
  unsigned char* arena = nullptr;
  CK(dalloc(ctx, (void**)&arena, total), "allocate tables");
  for (auto& t : small) {
    *t.first = arena;
    arena += (t.second + 255) / 256 * 256;
  }
  CK(dalloc(ctx, (void**)&ctx->staging, 2 * n * 2 * sizeof(double)), "allocate staging");
  CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), st), "clear error flag");

  // metric upload: the staging buffer holds the three fields during creation
  double* gdev[3] = {nullptr, nullptr, nullptr};
  for (int f = 0; f < 3; ++f) {
    if (g_host[f]) {
      gdev[f] = ctx->staging + (size_t)f * n;
      CK(cudaMemcpyAsync(gdev[f], g_host[f], n * sizeof(double), cudaMemcpyHostToDevice, st),
         "upload metric");
    }
  }
  // The log fields and their derivatives use psi/psiT-sized scratch in FP64.
  void *logs = nullptr, *logsT = nullptr, *dxT = nullptr, *dy = nullptr;
  CK(cudaMallocAsync(&logs, n * sizeof(Q4<double>), st), "allocate precompute scratch");
  CK(cudaMallocAsync(&logsT, n * sizeof(Q4<double>), st), "allocate precompute scratch");
  CK(cudaMallocAsync(&dxT, n * sizeof(Q4<double>), st), "allocate precompute scratch");
  CK(cudaMallocAsync(&dy, n * sizeof(Q4<double>), st), "allocate precompute scratch");
  CK(launch_metric_fields(gdev[0], gdev[1], gdev[2], (int)n, ctx->c, ctx->mass, ctx->conn,
                          ctx->a1, ctx->a2, ctx->meff, ctx->w, (Q4<double>*)logs, st),
     "metric fields");
  ctx->launches += 1;
  if (ctx->conn == DIRAC_CONN_NONE) {
    CK(cudaMemsetAsync(ctx->omx, 0, n * sizeof(double), st), "zero connection");
    CK(cudaMemsetAsync(ctx->omy, 0, n * sizeof(double), st), "zero connection");
  } else {
    // FP64 spectral derivatives with the same fused line pass (derivative mode)
    void *tx = nullptr, *ty = nullptr, *mx = nullptr, *my = nullptr;
    CK(cudaMallocAsync(&tx, nx * sizeof(Cx<double>), st), "allocate");
    CK(cudaMallocAsync(&ty, ny * sizeof(Cx<double>), st), "allocate");
    CK(cudaMallocAsync(&mx, nx * sizeof(Q4<double>), st), "allocate");
    CK(cudaMallocAsync(&my, ny * sizeof(Q4<double>), st), "allocate");
    const int sx = line_pass_radix_small<double>(nx, ny), sy = line_pass_radix_small<double>(ny, nx);
    CK(launch_twiddles<double>(nx, sx ? sx : line_pass_radix<double>(nx), (Cx<double>*)tx, st),
       "twiddles");
    CK(launch_twiddles<double>(ny, sy ? sy : line_pass_radix<double>(ny), (Cx<double>*)ty, st),
       "twiddles");
    CK(launch_deriv_mult<double>(nx, ctx->ax, (Q4<double>*)mx, st), "derivative table");
    CK(launch_deriv_mult<double>(ny, ctx->ay, (Q4<double>*)my, st), "derivative table");
    LinePassArgs<double> d{};
    d.L = nx; d.n_lines = ny; d.sigma = 0; d.tw = d.tw_small = (const Cx<double>*)tx;
    d.mult = (const Q4<double>*)mx; d.in = (const Q4<double>*)logs; d.out = (Q4<double>*)dxT;
    CK(launch_line_pass<double>(d, MODE_DERIV, 0, st), "x derivative of log fields");
    CK(launch_transpose<double>((const Q4<double>*)logs, (Q4<double>*)logsT, ny, nx, st),
       "transpose");
    d.L = ny; d.n_lines = nx; d.sigma = 1; d.tw = d.tw_small = (const Cx<double>*)ty;
    d.mult = (const Q4<double>*)my; d.in = (const Q4<double>*)logsT; d.out = (Q4<double>*)dy;
    CK(launch_line_pass<double>(d, MODE_DERIV, 0, st), "y derivative of log fields");
    const double fac = ctx->conn == DIRAC_CONN_PAPER_2D ? 0.25 : 0.5;
    CK(launch_omega((const Q4<double>*)dxT, (const Q4<double>*)dy, nx, ny, fac, ctx->omx,
                    ctx->omy, st),
       "spin connection");
    ctx->launches += 8;
    CK(cudaFreeAsync(tx, st), "free"); CK(cudaFreeAsync(ty, st), "free");
    CK(cudaFreeAsync(mx, st), "free"); CK(cudaFreeAsync(my, st), "free");
  }
  CK(cudaFreeAsync(logs, st), "free"); CK(cudaFreeAsync(logsT, st), "free");
  CK(cudaFreeAsync(dxT, st), "free"); CK(cudaFreeAsync(dy, st), "free");
  // absorbing layer and b - 1
  CK(launch_pml(nx, ctx->ax, ctx->abs.width_x, ctx->abs.type, ctx->abs.sigma0, ctx->abs.theta,
                ctx->sxinv, ctx->sxinv_im, st),
     "layer x");
  CK(launch_pml(ny, ctx->ay, ctx->abs.width_y, ctx->abs.type, ctx->abs.sigma0, ctx->abs.theta,
                ctx->syinv, ctx->syinv_im, st),
     "layer y");
  CK(launch_beta<T>(ctx->a1, ctx->a2, ctx->sxinv, ctx->syinv, ctx->sxinv_im, ctx->syinv_im, nx,
                    ny, (T*)ctx->beta1, (T*)ctx->beta2T, (T*)ctx->beta1_im,
                    (T*)ctx->beta2T_im, st),
     "b - 1");
  CK(launch_twiddles<T>(nx, line_pass_radix<T>(nx), (Cx<T>*)ctx->tw_x, st), "twiddles");
  CK(launch_twiddles<T>(ny, line_pass_radix<T>(ny), (Cx<T>*)ctx->tw_y, st), "twiddles");
  if (ctx->tw_x_alt)
    CK(launch_twiddles<T>(nx, line_pass_radix_alt<T>(nx), (Cx<T>*)ctx->tw_x_alt, st), "twiddles");
  if (ctx->tw_y_alt)
    CK(launch_twiddles<T>(ny, line_pass_radix_alt<T>(ny), (Cx<T>*)ctx->tw_y_alt, st), "twiddles");
  if (ctx->tw_x_small)
    CK(launch_twiddles<T>(nx, line_pass_radix_small<T>(nx, ny), (Cx<T>*)ctx->tw_x_small, st),
       "twiddles");
  if (ctx->tw_y_small)
    CK(launch_twiddles<T>(ny, line_pass_radix_small<T>(ny, nx), (Cx<T>*)ctx->tw_y_small, st),
       "twiddles");
  if (ctx->tw_x_team)
    CK(launch_team_twiddles<T>(nx, (Cx<T>*)ctx->tw_x_team, st), "twiddles");
  if (ctx->tw_y_team)
    CK(launch_team_twiddles<T>(ny, (Cx<T>*)ctx->tw_y_team, st), "twiddles");
  CK(launch_deriv_mult<T>(nx, ctx->ax, (Q4<T>*)ctx->dmult_x, st), "derivative table");
  CK(launch_deriv_mult<T>(ny, ctx->ay, (Q4<T>*)ctx->dmult_y, st), "derivative table");
  if (ctx->dmult_px)
    CK(launch_team_perm<T>(nx, (const Q4<T>*)ctx->dmult_x, (Q4<T>*)ctx->dmult_px, st),
       "multiplier order");
  if (ctx->dmult_py)
    CK(launch_team_perm<T>(ny, (const Q4<T>*)ctx->dmult_y, (Q4<T>*)ctx->dmult_py, st),
       "multiplier order");
  ctx->launches += 7;
  CK(cudaStreamSynchronize(st), "create");
  ctx->dt_cached = 0.0;
  return DIRAC_OK;
}

// ------------------------------------------------------------------ library-internal
dirac_status dgb_tables_for_dt(dirac_ctx* ctx, double dt) {
  return ctx->prec == DIRAC_C64 ? tables_for_dt<float>(ctx, dt) : tables_for_dt<double>(ctx, dt);
}

// Device bytes a context of this size holds at most (creation, state, half-step
// matrices, staging for host transfers, observables scratch and density).
size_t dgb_footprint_bytes(int nx, int ny, dirac_precision prec) {
  const size_t n = (size_t)nx * ny;
  const size_t r = prec == DIRAC_C64 ? 4 : 8, q4 = 4 * r;
  size_t per_point = 6 * sizeof(double)   // a1, a2, meff, w, omx, omy
                     + 2 * q4             // psi, psiT
                     + 2 * r              // b - 1 (both layouts)
                     + 3 * q4             // U (two layouts), U^2
                     + 4 * sizeof(double) // staging (complex128 spinor)
                     + 2 * q4             // observables scratch
                     + sizeof(double);    // density
  size_t per_line = (size_t)(nx + ny) * (sizeof(double) + 6 * q4);
  return n * per_point + per_line + 4 * sizeof(double) * 2048 + 4096;
}

// Times every CTA shape of one pass (reps launches each, CUDA events on the context's
// stream) with its output in scratch memory, so the state is untouched; returns the
// fastest shape (threads value for dirac_set_launch).
template <typename T>
static dirac_status tune_pass(dirac_ctx* ctx, int axis, int reps, int* best, float* best_ms) {
  LinePassArgs<T> a = pass_args<T>(ctx, axis);
  a.in = (const Q4<T>*)ctx->psi;  // any data of the pass's shape: the time does not depend on it
  a.out = (Q4<T>*)ctx->scratch1;
  a.mult = (const Q4<T>*)(axis == 0 ? ctx->mult_x : ctx->mult_y);
  a.mult_perm = (const Q4<T>*)(axis == 0 ? ctx->mult_px : ctx->mult_py);
  a.beta = (const T*)(axis == 0 ? ctx->beta1 : ctx->beta2T);
  a.u_store = (axis == 1 && !ctx->u_identity) ? (const Q4<T>*)ctx->u2_t : nullptr;
  const int L = a.L;
  const int options[5] = {256, 512, 1024, 256 | DIRAC_LAUNCH_ALT_RADIX,
                          512 | DIRAC_LAUNCH_ALT_RADIX};
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0), "tune");
  CK(cudaEventCreate(&e1), "tune");
  *best = 0;
  *best_ms = 1e30f;
  for (int t : options) {
    if (t == 1024 && !(sizeof(T) == 4 && L >= 256)) continue;  // team pass: complex64 only
    if ((t & DIRAC_LAUNCH_ALT_RADIX) && !line_pass_radix_alt<T>(L)) continue;
    const int opt = pass_opt(ctx, t, L, a.n_lines);
    cudaError_t e = cudaSuccess;
    for (int w = 0; w < 2 && e == cudaSuccess; ++w) e = launch_line_pass<T>(a, MODE_STEP, opt, ctx->stream);
    if (e == cudaSuccess) e = cudaEventRecord(e0, ctx->stream);
    for (int r = 0; r < reps && e == cudaSuccess; ++r) e = launch_line_pass<T>(a, MODE_STEP, opt, ctx->stream);
    if (e == cudaSuccess) e = cudaEventRecord(e1, ctx->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e != cudaSuccess) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      return cuda_fail(ctx, e, "autotune");
    }
    ctx->launches += reps + 2;
    if (ms < *best_ms) {
      *best_ms = ms;
      *best = t;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *best_ms /= reps;
  return DIRAC_OK;
}

template <typename T>
static dirac_status autotune_impl(dirac_ctx* ctx, int reps, int* tx, int* ty) {
  if (!ctx->scratch1) {
    CK(dalloc(ctx, &ctx->scratch1, npts(ctx) * sizeof(Q4<T>)), "scratch");
    CK(dalloc(ctx, &ctx->scratch2, npts(ctx) * sizeof(Q4<T>)), "scratch");
  }
  if (ctx->dt_cached == 0.0) {
    dirac_status s = tables_for_dt<T>(ctx, 0.01);
    if (s != DIRAC_OK) return s;
  }
  if (whole_steps(ctx, true)) {  // the default: whole steps in one launch, faster than any passes
    *tx = *ty = ctx->threads_x = ctx->threads_y = 0;
    return DIRAC_OK;
  }
  float mx, my;
  dirac_status s = tune_pass<T>(ctx, 0, reps, tx, &mx);
  if (s == DIRAC_OK) s = tune_pass<T>(ctx, 1, reps, ty, &my);
  if (s != DIRAC_OK) return s;
  ctx->threads_x = *tx;
  ctx->threads_y = *ty;
  return DIRAC_OK;
}

// ------------------------------------------------------------------------ the ABI
extern "C" {

dirac_status dirac_create(const dirac_grid* grid, const dirac_domain* domain,
                          const dirac_metric* metric, double mass, double c,
                          const dirac_absorber* absorber, dirac_precision precision,
                          void* cuda_stream, dirac_ctx** out) {
  if (!out) return fail(nullptr, DIRAC_EINVAL, "out is NULL");
  *out = nullptr;
  if (!grid || !domain) return fail(nullptr, DIRAC_EINVAL, "grid and domain are required");
  if (!pow2_in(grid->nx, 16, 4096) || !pow2_in(grid->ny, 16, 4096))
    return fail(nullptr, DIRAC_EINVAL, "nx and ny must be powers of two in [16, 4096]");
  if (!(domain->ax > 0.0) || !(domain->ay > 0.0) || !isfinite(domain->ax) || !isfinite(domain->ay))
    return fail(nullptr, DIRAC_EINVAL, "domain half-widths must be positive and finite");
  if (!(c > 0.0) || !isfinite(c) || !isfinite(mass))
    return fail(nullptr, DIRAC_EINVAL, "c must be positive and mass finite");
  if (precision != DIRAC_C64 && precision != DIRAC_C128)
    return fail(nullptr, DIRAC_EINVAL, "unknown precision");
  dirac_absorber ab = {0, 0, 1, 1.0, 0.0};
  if (absorber) {
    ab = *absorber;
    if (ab.width_x < 0 || ab.width_y < 0 || ab.width_x >= grid->nx / 2 ||
        ab.width_y >= grid->ny / 2)
      return fail(nullptr, DIRAC_EINVAL, "absorber widths must be in [0, N/2)");
    if ((ab.width_x > 0 || ab.width_y > 0) && (ab.type < 1 || ab.type > 6))
      return fail(nullptr, DIRAC_EINVAL, "absorber type must be 1..6");
    if (!isfinite(ab.sigma0) || ab.sigma0 < 0.0 || !isfinite(ab.theta))
      return fail(nullptr, DIRAC_EINVAL, "absorber sigma0 must be >= 0 and theta finite");
    if (ab.theta != 0.0 && (ab.width_x > 0 || ab.width_y > 0) && precision != DIRAC_C128)
      return fail(nullptr, DIRAC_EUNSUPPORTED,
                  "complex stretching (theta != 0) needs complex128 (a complex b)");
  }
  int conn = DIRAC_CONN_COVARIANT;
  const double* g_host[3] = {nullptr, nullptr, nullptr};
  if (metric) {
    conn = metric->conn;
    if (conn < 0 || conn > 2) return fail(nullptr, DIRAC_EINVAL, "unknown connection mode");
    g_host[0] = metric->g00;
    g_host[1] = metric->g11;
    g_host[2] = metric->g22;
    const size_t n = (size_t)grid->nx * grid->ny;
    for (int f = 0; f < 3; ++f) {
      if (!g_host[f]) continue;
      for (size_t k = 0; k < n; ++k) {
        const double v = g_host[f][k];
        if (!(v > 0.0) || !isfinite(v))
          return fail(nullptr, DIRAC_EINVAL, "metric entries must be positive and finite");
      }
    }
  }
  dirac_ctx* ctx = new (std::nothrow) dirac_ctx();
  if (!ctx) return fail(nullptr, DIRAC_ENOMEM, "host allocation failed");
  ctx->nx = grid->nx;
  ctx->ny = grid->ny;
  ctx->ax = domain->ax;
  ctx->ay = domain->ay;
  ctx->mass = mass;
  ctx->c = c;
  ctx->prec = precision;
  ctx->conn = conn;
  ctx->abs = ab;
  ctx->u_identity = (mass == 0.0 && conn == DIRAC_CONN_NONE);
  ctx->fault_alloc_at = fault_alloc_from_env();
  cudaGetDevice(&ctx->device);
  if (cuda_stream) {
    ctx->stream = (cudaStream_t)cuda_stream;
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      dirac_status s = cuda_fail(nullptr, e, "create stream");
      delete ctx;
      return s;
    }
    ctx->own_stream = true;
  }
  dirac_status s = precision == DIRAC_C64 ? create_impl<float>(ctx, g_host)
                                          : create_impl<double>(ctx, g_host);
  if (s != DIRAC_OK) {
    g_create_error = ctx->err;
    dirac_destroy(ctx);
    return s;
  }
  *out = ctx;
  return DIRAC_OK;
}

dirac_status dirac_set_state(dirac_ctx* ctx, const double* psi, int on_device) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (!psi) return fail(ctx, DIRAC_EINVAL, "psi is NULL");
  const size_t n = npts(ctx);
  const double* src = psi;
  if (!on_device) {
    CK(cudaMemcpyAsync(ctx->staging, psi, 4 * n * sizeof(double), cudaMemcpyHostToDevice,
                       ctx->stream),
       "upload state");
    src = ctx->staging;
  }
  if (ctx->prec == DIRAC_C64)
    CK(launch_pack<float>(src, (Q4<float>*)ctx->psi, n, ctx->stream), "pack state");
  else
    CK(launch_pack<double>(src, (Q4<double>*)ctx->psi, n, ctx->stream), "pack state");
  ctx->launches += 1;
  if (!on_device) CK(cudaStreamSynchronize(ctx->stream), "upload state");
  ctx->state_set = true;
  return DIRAC_OK;
}

dirac_status dirac_get_state(dirac_ctx* ctx, double* psi_out, int on_device) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (!psi_out) return fail(ctx, DIRAC_EINVAL, "psi_out is NULL");
  if (!ctx->state_set) return fail(ctx, DIRAC_ESTATE, "no state has been set");
  const size_t n = npts(ctx);
  double* dst = on_device ? psi_out : ctx->staging;
  if (ctx->prec == DIRAC_C64)
    CK(launch_unpack<float>((const Q4<float>*)ctx->psi, dst, n, ctx->stream), "unpack state");
  else
    CK(launch_unpack<double>((const Q4<double>*)ctx->psi, dst, n, ctx->stream), "unpack state");
  ctx->launches += 1;
  if (!on_device) {
    CK(cudaMemcpyAsync(psi_out, ctx->staging, 4 * n * sizeof(double), cudaMemcpyDeviceToHost,
                       ctx->stream),
       "download state");
    CK(cudaStreamSynchronize(ctx->stream), "download state");
    return device_error(ctx);
  }
  return DIRAC_OK;
}

dirac_status dirac_step(dirac_ctx* ctx, long n_steps, double dt) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (n_steps < 0) return fail(ctx, DIRAC_EINVAL, "n_steps must be >= 0");
  if (!(dt > 0.0) || !isfinite(dt)) return fail(ctx, DIRAC_EINVAL, "dt must be positive");
  if (!ctx->state_set) return fail(ctx, DIRAC_ESTATE, "set_state must come before step");
  if (n_steps == 0) return DIRAC_OK;
  return ctx->prec == DIRAC_C64 ? step_impl<float>(ctx, n_steps, dt)
                                : step_impl<double>(ctx, n_steps, dt);
}

dirac_status dirac_observables(dirac_ctx* ctx, dirac_obs* out, double* density_or_NULL) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (!out) return fail(ctx, DIRAC_EINVAL, "out is NULL");
  if (!ctx->state_set) return fail(ctx, DIRAC_ESTATE, "no state has been set");
  return ctx->prec == DIRAC_C64 ? observables_impl<float>(ctx, out, density_or_NULL)
                                : observables_impl<double>(ctx, out, density_or_NULL);
}

dirac_status dirac_synchronize(dirac_ctx* ctx) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  CK(cudaStreamSynchronize(ctx->stream), "synchronize");
  return device_error(ctx);
}

const char* dirac_last_error(const dirac_ctx* ctx) {
  return ctx ? ctx->err.c_str() : g_create_error.c_str();
}

void dirac_destroy(dirac_ctx* ctx) {
  if (!ctx) return;
  if (ctx->stream) cudaStreamSynchronize(ctx->stream);
  free_all(ctx);
  if (ctx->own_stream && ctx->stream) cudaStreamDestroy(ctx->stream);
  delete ctx;
}

dirac_status dirac_set_scheme(dirac_ctx* ctx, int scheme) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (scheme < DIRAC_SCHEME_II || scheme > DIRAC_SCHEME_CRANK_NICOLSON)
    return fail(ctx, DIRAC_EINVAL, "unknown scheme");
  if (scheme != ctx->scheme) {
    ctx->scheme = scheme;
    ctx->dt_cached = 0.0;  // the tables of the new order are made on the next step
  }
  return DIRAC_OK;
}

dirac_status dirac_set_potentials(dirac_ctx* ctx, const double* V, const double* Ax,
                                  const double* Ay) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  const size_t n = npts(ctx);
  const double* src[3] = {V, Ax, Ay};
  double** dst[3] = {&ctx->pot_v, &ctx->pot_ax, &ctx->pot_ay};
  for (int f = 0; f < 3; ++f)
    if (src[f])
      for (size_t k = 0; k < n; ++k)
        if (!isfinite(src[f][k])) return fail(ctx, DIRAC_EINVAL, "potentials must be finite");
  for (int f = 0; f < 3; ++f) {
    ctx->pot_use[f] = src[f] != nullptr;
    if (!src[f]) continue;  // an earlier buffer stays allocated for a later call
    if (!*dst[f]) {
      void* p = nullptr;
      if (dalloc(ctx, &p, n * sizeof(double)) != cudaSuccess)
        return fail(ctx, DIRAC_ENOMEM, "allocate potentials");
      *dst[f] = (double*)p;
    }
    cudaError_t e = cudaMemcpy(*dst[f], src[f], n * sizeof(double), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "copy potentials");
  }
  ctx->has_pot = V || Ax || Ay;
  ctx->dt_cached = 0.0;  // the half-step matrices are made again on the next step
  return DIRAC_OK;
}

dirac_status dirac_set_poly_degree(dirac_ctx* ctx, int degree) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (degree < 1 || degree > 256) return fail(ctx, DIRAC_EINVAL, "degree must be 1..256");
  ctx->poly_degree = degree;
  return DIRAC_OK;
}

dirac_status dirac_set_krylov(dirac_ctx* ctx, double tol, int restart, int max_restarts) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (!(tol >= 0.0) || !isfinite(tol) || restart < 1 || restart > 100 || max_restarts < 0)
    return fail(ctx, DIRAC_EINVAL, "tol >= 0, restart in 1..100, max_restarts >= 0");
  ctx->krylov_tol = tol;
  ctx->krylov_m = restart;
  ctx->krylov_restarts = max_restarts;
  return DIRAC_OK;
}

long dirac_krylov_iterations(const dirac_ctx* ctx) { return ctx ? ctx->krylov_iters : 0; }

dirac_status dirac_set_launch(dirac_ctx* ctx, int threads_x_pass, int threads_y_pass) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  const int t[2] = {threads_x_pass, threads_y_pass};
  for (int k = 0; k < 2; ++k) {
    const int th = t[k] & ~DIRAC_LAUNCH_ALT_RADIX;
    const bool alt = (t[k] & DIRAC_LAUNCH_ALT_RADIX) != 0;
    if ((th != 0 && th != 256 && th != 512 && th != 1024) || (alt && th != 256 && th != 512))
      return fail(ctx, DIRAC_EINVAL,
                  "shape must be 0 (default), 256, 512 or 1024, or 256 or 512 plus "
                  "DIRAC_LAUNCH_ALT_RADIX");
  }
  ctx->threads_x = threads_x_pass;
  ctx->threads_y = threads_y_pass;
  return DIRAC_OK;
}

long dirac_launch_count(const dirac_ctx* ctx) { return ctx ? ctx->launches : 0; }

dirac_status dirac_test_timeout_next_step(dirac_ctx* ctx) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  ctx->test_timeout_next = 16;
  return DIRAC_OK;
}

dirac_status dirac_autotune(dirac_ctx* ctx, int reps, int* threads_x, int* threads_y) {
  if (!ctx) return fail(nullptr, DIRAC_EINVAL, "ctx is NULL");
  if (!threads_x || !threads_y || reps < 1) return fail(ctx, DIRAC_EINVAL, "bad arguments");
  if (!ctx->state_set) return fail(ctx, DIRAC_ESTATE, "set_state must come before autotune");
  return ctx->prec == DIRAC_C64 ? autotune_impl<float>(ctx, reps, threads_x, threads_y)
                                : autotune_impl<double>(ctx, reps, threads_x, threads_y);
}

size_t dirac_footprint_bytes(const dirac_grid* grid, dirac_precision precision) {
  if (!grid || grid->nx <= 0 || grid->ny <= 0) return 0;
  return dgb_footprint_bytes(grid->nx, grid->ny, precision);
}

}  // extern "C"
