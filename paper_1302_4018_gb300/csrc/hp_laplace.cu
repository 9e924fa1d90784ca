// Shifted periodic Laplacian (the control problem of Section 5):
//   (A x)(s) = (8 + m + mu(s)) x(s) - sum_mu [x(s + mu) + x(s - mu)]
// in FP64, and multi-right-hand-side CG for the quadratures v^H A^-1 v.
// A is real, so a complex probe is solved as two real right-hand sides
// (its real and imaginary parts); the cross terms of v^H x cancel because
// A is symmetric.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "hp_internal.h"

static int lblocks(hp_ctx* ctx, long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  long long cap = (long long)ctx->num_sms * 16;
  return (int)std::max(1LL, std::min(b, cap));
}

// The diagonal as the stencil below uses it: 8 + m + mu(s), less 2 for every extent of 1 (there both neighbours are the
// site itself).  FP64 adds bound the stencil (2 lanes per clock and SM), so a 3-D lattice padded to four dimensions does
// not add its own site twice.
__device__ __forceinline__ double lap_diag0(const LatGeom& g) {
  double d = 8.0 + g.mass;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (g.L[j] == 1) d -= 2.0;
  return d;
}

// MF: a per-site mass field (a branch per site would add it on the FP64 pipe either way); NC: x is not written while the
// kernel runs (read-only loads)
template <bool MF, bool NC = true>
__device__ __forceinline__ double lap_site(const LatGeom& g, double diag0, const double* x, int site) {
  auto ld = [x](int i) { return NC ? __ldg(x + i) : x[i]; };
  int r = site, st = 1;
  double acc = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int L = g.L[j];
    if (L == 1) continue;   // uniform over the grid
    const int xj = r % L;
    r /= L;
    const int fw = (xj + 1 == L) ? site - (L - 1) * st : site + st;
    const int bw = (xj == 0) ? site + (L - 1) * st : site - st;
    const double t = ld(fw) + ld(bw);
    acc = j == 0 ? t : acc + t;
    st *= L;
  }
  const double diag = MF ? diag0 + g.mass_field[site] : diag0;
  return fma(diag, ld(site), -acc);
}

__global__ void k_lap_apply(LatGeom g, const double* __restrict__ in, double* __restrict__ out, int nrhs) {
  const long long total = (long long)nrhs * g.V;
  const double diag0 = lap_diag0(g);
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int rhs = (int)(t / g.V), site = (int)(t - (long long)rhs * g.V);
    const double* x = in + (size_t)rhs * g.V;
    out[t] = g.mass_field ? lap_site<true>(g, diag0, x, site) : lap_site<false>(g, diag0, x, site);
  }
}

hp_status hp_apply_laplace(hp_ctx* ctx, LatGeom g, int nrhs, const double* in, double* out) {
  const size_t bytes = sizeof(double) * (size_t)nrhs * g.V;
  const void* din = nullptr;
  HP_TRY(hp_device_view(ctx, in, bytes, "apply.lap_in", &din));
  double* dout = out;
  bool out_host = !hp_is_device_ptr(out);
  if (out_host) {
    void* p = nullptr;
    HP_TRY(hp_ws(ctx, "apply.lap_out", bytes, &p));
    dout = (double*)p;
  }
  {
    ProfScope ps(ctx, "k_lap_apply");
    k_lap_apply<<<lblocks(ctx, (long long)nrhs * g.V, 256), 256, 0, ctx->stream>>>(g, (const double*)din, dout, nrhs);
  }
  HP_LAUNCH_CHECK();
  if (out_host) {
    HP_CUDA(cudaMemcpyAsync(out, dout, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    HP_CUDA(cudaStreamSynchronize(ctx->stream));
  }
  return HP_OK;
}

// ------------------------------------------------------------------ CG kernels
struct LArgs {
  const LatGeom* lats;
  SlotState* st;
  double* part;
  unsigned int* cnt;
  int Vmax, gy;
  double *x, *r, *p, *q;   // [slot][Vmax]
  double tol2;
  int maxiter;
  int nslots;
  double* dc;    // deflation: V^T b of each slot's source, [slot][defl_k]
};

#define LSLOT(COND)                                                \
  const int slot = blockIdx.x, bx = blockIdx.y, gx = gridDim.y;    \
  SlotState* S = a.st + slot;                                      \
  if (!(COND)) return;                                             \
  const LatGeom g = a.lats[S->lat];                                \
  const int ntiles = (g.V + NT - 1) / NT;                          \
  if (bx >= ntiles) return;                                        \
  const int nparts = min(gx, ntiles);                              \
  double* part = a.part + (size_t)slot * 4 * a.gy;                 \
  const size_t off = (size_t)slot * a.Vmax;                        \
  (void)nparts;                                                    \
  (void)part;

__device__ __forceinline__ double lap_source(const LatGeom& g, int site, int m, int part) {
  double2 v = g.ptab[probe_phase(g, (uint32_t)site, (uint32_t)m)];
  return part == 0 ? v.x : v.y;
}

// the solved source: the probe, projected off the deflated eigenvectors when there are any
__device__ __forceinline__ double lap_src(const LatGeom& g, const LArgs& a, int slot, int site, int m, int part) {
  double b = lap_source(g, site, m, part);
  if (g.defl_k) {
    const double* c = a.dc + (size_t)slot * g.defl_k;
    for (int j = 0; j < g.defl_k; ++j) b -= c[j] * g.defl_V[(size_t)j * g.V + site];
  }
  return b;
}

// deflation coefficients c_j = V_j^T b of the slots being filled: block (j, slot), one sum over
// the lattice in a fixed order
template <int NT>
__global__ void __launch_bounds__(NT) k_cg_defl(LArgs a) {
  const int j = blockIdx.x, slot = blockIdx.y;
  const SlotState* S = a.st + slot;
  if (S->status != SLOT_INIT) return;
  const LatGeom g = a.lats[S->lat];
  if (j >= g.defl_k) return;
  double acc[1] = {0.0};
  const double* vj = g.defl_V + (size_t)j * g.V;
  for (int site = threadIdx.x; site < g.V; site += NT) acc[0] += vj[site] * lap_source(g, site, S->m, S->a);
  __shared__ double sh[NT / 32];
  double t = acc[0];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < NT / 32; ++w) tot += sh[w];
    a.dc[(size_t)slot * g.defl_k + j] = tot;
  }
}

// Block sum of v into part[q * gy + bx].  One warp adds the block's values (NT / 32 per lane, then a shuffle tree):
// NT / 32 + 5 FP64 warp instructions a block, where a shuffle tree in every warp takes 5 NT / 32 and FP64 runs at 2
// lanes per clock (8^4, 256 slots: a k_cg_xr launch 22.7 -> 19.9 us).
template <int NQ, int NT>
__device__ __forceinline__ void lreduce(double (&v)[NQ], double* part, int gy, int bx) {
  __shared__ double sh[NQ][NT];
#pragma unroll
  for (int qq = 0; qq < NQ; ++qq) sh[qq][threadIdx.x] = v[qq];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int qq = 0; qq < NQ; ++qq) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < NT / 32; w += 2) t += sh[qq][threadIdx.x + 32 * w] + sh[qq][threadIdx.x + 32 * w + 32];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (threadIdx.x == 0) part[(size_t)qq * gy + bx] = t;
    }
  }
}

// ---- per-slot scalar steps of CG (one thread, after the slot's reduction): shared by the
// lattice engine (one slot per block row) and the blocked sparse engine (all slots per block)
__device__ __forceinline__ void cg_after_init(SlotState* S, const LatGeom& g, double bb) {
  S->bnorm2 = bb;
  S->rnorm2 = bb;
  S->rmax2 = bb;
  S->rho = make_double2(bb, 0.0);
  S->iters = 0;
  S->updates = 0;
  S->need_update = 0;
  S->restart = 0;
  S->true_res2 = bb;
  S->gauss = 0.0;
  S->radau = g.quad_mu > 0.0 ? 1.0 / g.quad_mu : 0.0;
  S->status = bb > 0.0 ? SLOT_RUN : SLOT_DONE;
}

// alpha = rr / (p, A p)
__device__ __forceinline__ void cg_after_ap(SlotState* S, double pq) {
  S->alpha = make_double2(pq != 0.0 ? S->rho.x / pq : 0.0, 0.0);
  S->gauss += S->alpha.x * S->rho.x;   // Gauss rule: G_{k+1} = G_k + gamma_k ||r_k||^2
  S->restart = 0;
  S->sloppy_mv += 1;
}

// beta = rr' / rr, the Gauss-Radau coefficient, and the stopping tests
// delta2 > 0 (mixed precision): also ask for a true residual once ||r||^2 fell below delta2 times
// its largest value since the last one (reliable updates)
__device__ __forceinline__ void cg_after_xr(SlotState* S, const LatGeom& g, double rr, double tol2, int maxiter,
                                            double delta2 = 0.0) {
  const double delta = S->rho.x != 0.0 ? rr / S->rho.x : 0.0;
  S->beta = make_double2(delta, 0.0);
  S->rho = make_double2(rr, 0.0);
  S->rnorm2 = rr;
  S->rmax2 = fmax(S->rmax2, rr);
  S->iters += 1;
  if (g.quad_mu > 0.0) {   // Gauss-Radau: gt_{k+1} = (gt_k - gamma_k) / (mu (gt_k - gamma_k) + delta_{k+1})
    const double d = S->radau - S->alpha.x;
    const double den = g.quad_mu * d + delta;
    S->radau = den > 0.0 ? fmax(d, 0.0) / den : 0.0;
  }
  if (S->iters >= maxiter) {
    S->status = SLOT_FAIL;
    S->need_update = 1;
  } else if (g.quad_tol > 0.0) {   // stop on the quadrature bracket: no residual test, no restart
    if (S->radau * rr <= g.quad_tol * S->gauss || rr == 0.0 || !(rr == rr)) {
      S->true_res2 = rr;
      S->status = (rr == rr) ? SLOT_DONE : SLOT_FAIL;
    }
  } else if (rr <= tol2 * S->bnorm2 || !(rr == rr) || rr <= delta2 * S->rmax2) {
    S->need_update = 1;
  }
}

// the FP64 true residual: converged, or continue from it with p = r (keep_p: with the old p,
// the reliable update of mixed precision)
__device__ __forceinline__ void cg_after_true(SlotState* S, double rr, double tol2, bool keep_p = false) {
  S->true_res2 = rr;
  S->updates += 1;
  S->fp64_mv += 1;
  S->need_update = 0;
  if (S->status == SLOT_RUN) {
    if (rr <= tol2 * S->bnorm2) {
      S->status = SLOT_DONE;
    } else {
      S->rho = make_double2(rr, 0.0);
      S->rnorm2 = rr;
      S->rmax2 = rr;
      S->restart = keep_p ? 0 : 1;
    }
  }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_cg_init(LArgs a) {
  LSLOT(S->status == SLOT_INIT)
  double acc[1] = {0.0};
  const int m = S->m, pa = S->a;
  for (int tile = bx; tile < ntiles; tile += gx) {
    const int site = tile * NT + threadIdx.x;
    if (site >= g.V) continue;
    double b = lap_src(g, a, slot, site, m, pa);
    a.x[off + site] = 0.0;
    a.r[off + site] = b;
    a.p[off + site] = b;
    acc[0] += b * b;
  }
  lreduce<1, NT>(acc, part, a.gy, bx);
  if (last_block(a.cnt + slot, nparts)) {
    double tot[1];
    block_sum_partials<1, NT>(part, a.gy, nparts, tot);
    if (threadIdx.x == 0) {
      cg_after_init(S, g, tot[0]);
      a.cnt[slot] = 0;
    }
  }
}

// Sites of a block: tiles bx, bx + gx, ..., U of them per step, so that a thread has U independent sets of loads (and
// of FP64 chains) in flight.
#define LTILES(U) for (int tile = bx; tile < ntiles; tile += (U) * gx)
#define LSITE(u) const int site = (tile + (u) * gx) * NT + (int)threadIdx.x

// q = A p ; alpha = rr / (p, q).  Bound by the FP64 pipe (5 or 7 adds, 2 FMAs a site: 47 us for 16 slots of 64^3).
template <int NT, bool MF>
__device__ __forceinline__ double cg_ap_sites(const LatGeom& g, const double* __restrict__ p, double* __restrict__ q,
                                              int bx, int gx, int ntiles) {
  const double diag0 = lap_diag0(g);
  double acc = 0.0;
  LTILES(2) {
    double qv[2], pv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      LSITE(u);
      qv[u] = pv[u] = 0.0;
      if (site >= g.V) continue;
      qv[u] = lap_site<MF>(g, diag0, p, site);
      pv[u] = __ldg(p + site);
      q[site] = qv[u];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) acc = fma(pv[u], qv[u], acc);
  }
  return acc;
}
template <int NT>
__global__ void __launch_bounds__(NT) k_cg_ap(LArgs a) {
  LSLOT(S->status == SLOT_RUN)
  double acc[1] = {g.mass_field ? cg_ap_sites<NT, true>(g, a.p + off, a.q + off, bx, gx, ntiles)
                                : cg_ap_sites<NT, false>(g, a.p + off, a.q + off, bx, gx, ntiles)};
  lreduce<1, NT>(acc, part, a.gy, bx);
  if (last_block(a.cnt + slot, nparts)) {
    double tot[1];
    block_sum_partials<1, NT>(part, a.gy, nparts, tot);
    if (threadIdx.x == 0) {
      cg_after_ap(S, tot[0]);
      a.cnt[slot] = 0;
    }
  }
}

// x += alpha p ; r -= alpha q ; beta = rr' / rr
template <int NT>
__global__ void __launch_bounds__(NT) k_cg_xr(LArgs a) {
  LSLOT(S->status == SLOT_RUN)
  const double al = S->alpha.x;
  double acc[1] = {0.0};
  double* __restrict__ x = a.x + off;
  double* __restrict__ r = a.r + off;
  const double* __restrict__ p = a.p + off;
  const double* __restrict__ q = a.q + off;
  LTILES(2) {
    double xv[2], pv[2], rv[2], qv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      LSITE(u);
      if (site >= g.V) continue;
      xv[u] = x[site];
      pv[u] = p[site];
      rv[u] = r[site];
      qv[u] = q[site];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      LSITE(u);
      if (site >= g.V) continue;
      x[site] = fma(al, pv[u], xv[u]);
      const double rn = fma(-al, qv[u], rv[u]);
      r[site] = rn;
      acc[0] = fma(rn, rn, acc[0]);
    }
  }
  lreduce<1, NT>(acc, part, a.gy, bx);
  if (last_block(a.cnt + slot, nparts)) {
    double tot[1];
    block_sum_partials<1, NT>(part, a.gy, nparts, tot);
    if (threadIdx.x == 0) {
      cg_after_xr(S, g, tot[0], a.tol2, a.maxiter);
      a.cnt[slot] = 0;
    }
  }
}

// true residual r = b - A x.  Most iterations no slot asks for one: the grid is (1, tiles, classes) and block z
// loops over the slots z, z + gz, ... that ask (a slot is finalised by the last block that serves it, so all of them
// read its flag before); a block per (slot, tile) cost 10-12 us per idle launch.
template <int NT>
__global__ void __launch_bounds__(NT) k_cg_true(LArgs a) {
  __shared__ unsigned int want;
  // the flags of up to 32 of the block's slots at a time, one per lane
  for (int s0 = blockIdx.z; s0 < a.nslots; s0 += 32 * gridDim.z) {
   __syncthreads();
   if (threadIdx.x < 32) {
    const int sl = s0 + (int)threadIdx.x * gridDim.z;
    const unsigned int b = __ballot_sync(0xffffffffu, sl < a.nslots && a.st[min(sl, a.nslots - 1)].need_update);
    if (threadIdx.x == 0) want = b;
   }
   __syncthreads();
   for (unsigned int todo = want; todo; todo &= todo - 1) {
    const int slot = s0 + (__ffs(todo) - 1) * gridDim.z;
    SlotState* S = a.st + slot;
    const LatGeom g = a.lats[S->lat];
    const int ntiles = (g.V + NT - 1) / NT, bx = blockIdx.y, gx = gridDim.y;
    if (bx >= ntiles) continue;
    const int nparts = min(gx, ntiles);
    double* part = a.part + (size_t)slot * 4 * a.gy;
    const size_t off = (size_t)slot * a.Vmax;
    const double diag0 = lap_diag0(g);
    double acc[1] = {0.0};
    const int m = S->m, pa = S->a;
    for (int tile = bx; tile < ntiles; tile += gx) {
      const int site = tile * NT + threadIdx.x;
      if (site >= g.V) continue;
      const double ax = g.mass_field ? lap_site<true>(g, diag0, a.x + off, site) : lap_site<false>(g, diag0, a.x + off, site);
      const double rv = lap_src(g, a, slot, site, m, pa) - ax;
      a.r[off + site] = rv;
      acc[0] += rv * rv;
    }
    lreduce<1, NT>(acc, part, a.gy, bx);
    if (last_block(a.cnt + slot, nparts)) {
      double tot[1];
      block_sum_partials<1, NT>(part, a.gy, nparts, tot);
      if (threadIdx.x == 0) {
        cg_after_true(S, tot[0], a.tol2);
        a.cnt[slot] = 0;
      }
    }
   }
  }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_cg_p(LArgs a) {
  LSLOT(S->status == SLOT_RUN)
  const double be = S->restart ? 0.0 : S->beta.x;
  double* __restrict__ p = a.p + off;
  const double* __restrict__ r = a.r + off;
  LTILES(4) {
    double pv[4], rv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      LSITE(u);
      if (site >= g.V) continue;
      pv[u] = p[site];
      rv[u] = r[site];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      LSITE(u);
      if (site < g.V) p[site] = fma(be, pv[u], rv[u]);
    }
  }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_lquad(LArgs a) {
  LSLOT(S->status == SLOT_DONE || S->status == SLOT_FAIL)
  double acc[1] = {0.0};
  const int m = S->m, pa = S->a;
  for (int tile = bx; tile < ntiles; tile += gx) {
    const int site = tile * NT + threadIdx.x;
    if (site >= g.V) continue;
    acc[0] += lap_src(g, a, slot, site, m, pa) * a.x[off + site];
  }
  lreduce<1, NT>(acc, part, a.gy, bx);
  if (last_block(a.cnt + slot, nparts)) {
    double tot[1];
    block_sum_partials<1, NT>(part, a.gy, nparts, tot);
    if (threadIdx.x == 0) {
      S->q = make_double2(tot[0], 0.0);
      a.cnt[slot] = 0;
    }
  }
}

// g(site) += x(site)^2 over harvested slots of one lattice (A real symmetric: A^-H v = x)
__global__ void k_lgrad(LArgs a, int lat, const int* __restrict__ slots, int nsl, double* __restrict__ grad, int V) {
  for (int site = blockIdx.x * blockDim.x + threadIdx.x; site < V; site += gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int i = 0; i < nsl; ++i) {
      const int slot = slots[i];
      if (a.st[slot].lat != lat) continue;
      double xv = a.x[(size_t)slot * a.Vmax + site];
      acc += xv * xv;
    }
    grad[site] += acc;
  }
}

struct LaplaceEngine {
  static constexpr int NT = 256;
  static constexpr int LAP_BLOCKS = 6;   // resident blocks per SM
  int kernels_per_iteration() const { return 4; }
  static constexpr int GROUP_MAX = 1;
  hp_ctx* ctx;
  LArgs a;
  int nslots, gy, gy_true, gz_true;
  int big_lat = 0;   // index of the largest lattice (set by the scheduler; unused here)
  bool one_lat = false;   // one lattice in the problem (set by the scheduler; unused here)
  int defl_k = 0;
  dim3 grid() const { return dim3(nslots, gy); }
  // 4M sites' worth of slots: 128^2x64 with 32 vectors took 116 ms in 12 slots, 122 in 32
  static constexpr bool MORE_SLOTS = false;
  int group() const { return 1; }
  hp_status setup(int ns, int Vmax, const LatGeom* lats_dev, SlotState* st, const hp_solver_opts& o, double tol,
                  double, const LatGeom& big) {
    nslots = ns;
    memset(&a, 0, sizeof(a));
    a.lats = lats_dev;
    a.st = st;
    a.Vmax = Vmax;
    a.nslots = ns;
    // one resident wave over all slots: a thread then sums several sites before the block's FP64 shuffle sums (ten
    // adds per warp, as much as the stencil of one site) and a slot has few partial sums
    const int ntiles = (Vmax + NT - 1) / NT;
    gy = std::max(1, std::min(ntiles, (ctx->num_sms * LAP_BLOCKS + ns - 1) / ns));
    gy_true = std::max(1, std::min(ntiles, ctx->num_sms * 2));
    gz_true = std::max(1, std::min({ns, ctx->num_sms * LAP_BLOCKS / gy_true, 64}));
    a.gy = std::max(gy, gy_true);
    void* p = nullptr;
    HP_TRY(hp_ws(ctx, "solve.part", sizeof(double) * 4 * (size_t)ns * a.gy, &p));
    a.part = (double*)p;
    HP_TRY(hp_ws(ctx, "solve.cnt", sizeof(unsigned int) * ns, &p));
    a.cnt = (unsigned int*)p;
    HP_CUDA(cudaMemsetAsync(a.cnt, 0, sizeof(unsigned int) * ns, ctx->stream));
    const size_t fb = sizeof(double) * (size_t)ns * Vmax;
    HP_TRY(hp_ws(ctx, "solve.lx", fb, &p));
    a.x = (double*)p;
    HP_TRY(hp_ws(ctx, "solve.lr", fb, &p));
    a.r = (double*)p;
    HP_TRY(hp_ws(ctx, "solve.lp", fb, &p));
    a.p = (double*)p;
    HP_TRY(hp_ws(ctx, "solve.lq", fb, &p));
    a.q = (double*)p;
    a.tol2 = tol * tol;
    a.maxiter = o.maxiter > 0 ? o.maxiter : 10000;
    defl_k = big.defl_k;
    if (defl_k) {
      HP_TRY(hp_ws(ctx, "solve.defl_c", sizeof(double) * (size_t)ns * defl_k, &p));
      a.dc = (double*)p;
    }
    return HP_OK;
  }
  hp_status init() {
    if (defl_k) {
      ProfScope ps(ctx, "k_cg_defl");
      k_cg_defl<NT><<<dim3(defl_k, nslots), NT, 0, ctx->stream>>>(a);
    }
    {
      ProfScope ps(ctx, "k_cg_init");
      k_cg_init<NT><<<grid(), NT, 0, ctx->stream>>>(a);
    }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
  hp_status iteration() {
    { ProfScope ps(ctx, "k_cg_ap"); k_cg_ap<NT><<<grid(), NT, 0, ctx->stream>>>(a); }
    { ProfScope ps(ctx, "k_cg_xr"); k_cg_xr<NT><<<grid(), NT, 0, ctx->stream>>>(a); }
    { ProfScope ps(ctx, "k_cg_true"); k_cg_true<NT><<<dim3(1, gy_true, gz_true), NT, 0, ctx->stream>>>(a); }
    { ProfScope ps(ctx, "k_cg_p"); k_cg_p<NT><<<grid(), NT, 0, ctx->stream>>>(a); }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
  hp_status keep(const std::vector<int>&, const std::vector<SlotState>&, const SolveProblem&) {
    hp_set_error("solutions are kept for the Wilson operator only");
    return HP_EUNSUPPORTED;
  }
  hp_status harvest(const std::vector<int>& done_slots, const SolveProblem& pb, int* dev_slots) {
    {
      ProfScope ps(ctx, "k_lquad");
      k_lquad<NT><<<grid(), NT, 0, ctx->stream>>>(a);
    }
    HP_LAUNCH_CHECK();
    if (pb.want_grad && !done_slots.empty()) {
      HP_CUDA(cudaMemcpyAsync(dev_slots, done_slots.data(), sizeof(int) * done_slots.size(), cudaMemcpyHostToDevice,
                              ctx->stream));
      for (size_t L = 0; L < pb.lats.size(); ++L) {
        ProfScope ps(ctx, "k_lgrad");
        k_lgrad<<<lblocks(ctx, pb.lats[L].V, 256), 256, 0, ctx->stream>>>(a, (int)L, dev_slots, (int)done_slots.size(),
                                                                          pb.grad_dev[L], pb.lats[L].V);
      }
      HP_LAUNCH_CHECK();
    }
    return HP_OK;
  }
};

// ------------------------------------------------------------ blocked sparse CG
// A general sparse matrix runs all B = 32 SPL slots as one block of vectors laid out
// [row][slot] (lane l of a warp owns the slots l SPL .. l SPL + SPL - 1).  One warp per row reads the row's
// CSR entries once for every slot and gathers B contiguous values per entry (whole sectors), where one slot
// per block row would re-read the matrix for every slot and gather single words.  Reductions: each block
// leaves its sum per slot, the last block of 32 adds theirs, the last of those adds the groups' sums in
// a fixed order and takes the scalar CG steps of every slot.
struct BArgs {
  const LatGeom* lat;
  SlotState* st;
  double *x, *r, *p, *q;   // [n][B]
  double* part;            // [blocks][B]
  double* gpart;           // [groups of 32 blocks][B]
  unsigned int* cnt;       // per reducing kernel: one counter, then one per group
  int ngroups_max;
  int nblk;               // blocks of the matrix-vector kernels
  int nstream;            // blocks of the streaming kernels
  double tol2;
  int maxiter;
  // mixed precision: r, p, q and the correction xl in FP32, x = xh + xl with xh in FP64
  float *xl, *rf, *pf, *qf;
  const float* val32;     // the CSR values rounded to FP32
  double delta2;          // reliable-update threshold (squared)
};

enum { BK_INIT = 0, BK_AP, BK_XR, BK_TRUE, BK_QUAD, BK_COUNT };
constexpr int BT = 256;   // threads per block of the blocked kernels

__device__ __forceinline__ bool bk_on(const SlotState* S, int kind) {
  switch (kind) {
    case BK_INIT: return S->status == SLOT_INIT;
    case BK_AP:
    case BK_XR: return S->status == SLOT_RUN;
    case BK_TRUE: return S->need_update != 0;
    default: return S->status == SLOT_DONE || S->status == SLOT_FAIL;
  }
}

// N neighbouring slots of a row, moved in 16-byte pieces
template <typename T, int N>
struct alignas(sizeof(T) * N > 16 ? 16 : sizeof(T) * N) Pack {
  T v[N];
};

// t: the block's sum of slot threadIdx.x (threads < B).  The FP64 additions of one block over all partial sums (64 slots
// x 1216 blocks: 2400 warp instructions at 16 cycles, 20 us at the end of every launch) run in groups side by side.
template <int B>
__device__ __forceinline__ void bk_finish(const BArgs& a, const LatGeom& g, int kind, double t) {
  __shared__ int am_last;
  const int nb = gridDim.x, grp = blockIdx.x >> 5, ng = (nb + 31) >> 5, members = min(32, nb - 32 * grp);
  unsigned int* cnt = a.cnt + kind * (1 + a.ngroups_max);
  if (threadIdx.x < B) a.part[(size_t)blockIdx.x * B + threadIdx.x] = t;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = atomicAdd(cnt + 1 + grp, 1u) == (unsigned)members - 1u;
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  if (threadIdx.x < B) {
    const double* ps = a.part + (size_t)32 * grp * B + threadIdx.x;
    t = 0.0;
#pragma unroll 8
    for (int k = 0; k < members; ++k) t += __ldcg(ps + (size_t)k * B);
    a.gpart[(size_t)grp * B + threadIdx.x] = t;
  }
  if (threadIdx.x == 0) cnt[1 + grp] = 0;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = atomicAdd(cnt, 1u) == (unsigned)ng - 1u;
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  if (threadIdx.x < B) {
    double tot = 0.0;
#pragma unroll 8
    for (int k = 0; k < ng; ++k) tot += __ldcg(a.gpart + (size_t)k * B + threadIdx.x);
    SlotState* S = a.st + threadIdx.x;
    if (bk_on(S, kind)) {
      switch (kind) {
        case BK_INIT: cg_after_init(S, g, tot); break;
        case BK_AP: cg_after_ap(S, tot); break;
        case BK_XR: cg_after_xr(S, g, tot, a.tol2, a.maxiter, a.delta2); break;
        default: S->q = make_double2(tot, 0.0); break;
      }
    }
  }
  if (threadIdx.x == 0) *cnt = 0;
}

// the block's sum of slot threadIdx.x (threads < 32 SPL) from the lanes' sums of the slots they own
template <int SPL, typename T>
__device__ __forceinline__ double bk_sum_lanes(const T (&acc)[SPL]) {
  constexpr int B = 32 * SPL, NW = BT / 32;
  __shared__ T sh[NW][B];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < SPL; ++k) sh[warp][lane * SPL + k] = acc[k];
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < B)
#pragma unroll
    for (int w = 0; w < NW; ++w) t += (double)sh[w][threadIdx.x];
  return t;
}
// the same for the streaming kernels, where thread t holds the sums of the VW slots from (t % (B / VW)) VW on
template <int B, int VW, typename T>
__device__ __forceinline__ double bk_sum_cols(const T (&acc)[VW]) {
  constexpr int TPR = B / VW;
  __shared__ T sh[BT / TPR][B];
#pragma unroll
  for (int k = 0; k < VW; ++k) sh[threadIdx.x / TPR][(threadIdx.x % TPR) * VW + k] = acc[k];
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < B)
#pragma unroll
    for (int w = 0; w < BT / TPR; ++w) t += (double)sh[w][threadIdx.x];
  return t;
}

#define BK_ROWS(i) for (int i = blockIdx.x * (BT / 32) + (threadIdx.x >> 5); i < g.V; i += gridDim.x * (BT / 32))

// x = 0, r = p = b for the slots being filled; ||b||^2  (MIXED: r, p and the correction in FP32)
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(BT) k_bcg_init(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  int m[SPL], pa[SPL];
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane * SPL + k;
    on[k] = bk_on(S, BK_INIT);
    m[k] = S->m;
    pa[k] = S->a;
    acc[k] = 0.0;
  }
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      const size_t o = (size_t)i * B + lane * SPL + k;
      const double b = lap_source(g, i, m[k], pa[k]);
      a.x[o] = 0.0;
      if (MIXED) {
        a.xl[o] = 0.0f;
        a.rf[o] = (float)b;
        a.pf[o] = (float)b;
      } else {
        a.r[o] = b;
        a.p[o] = b;
      }
      acc[k] += b * b;
    }
  }
  bk_finish<B>(a, g, BK_INIT, bk_sum_lanes<SPL>(acc));
}

// q = A p, (p, q): in FP64, or (MIXED) in FP32 with the block sums in FP64.
// A warp walks rows gw, gw + tw, ...: the row pointers two rows ahead and the entries one row ahead are requested before the
// gathers of the current row, so a row costs the warp one memory latency (its gathers, eight at a time in flight), and
// the resident warps cover it.  A walk over contiguous rows of one entry stream, flushing rows as they ended, spent
// 153 us where this takes 87 (64^3 grid renumbered, B = 64, FP32; 134 MB of p and q plus 470 MB of gathers from L2).
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(BT, SPL == 4 ? (MIXED ? 4 : 2) : 4) k_bcg_ap(BArgs a) {
  typedef typename std::conditional<MIXED, float, double>::type T;
  typedef Pack<T, SPL> P;
  constexpr int B = 32 * SPL, U = sizeof(P) >= 16 ? 4 : 8;
  constexpr unsigned FULL = 0xffffffffu;
  const LatGeom& g = *a.lat;   // by reference: a copy of the struct costs 20 registers
  const int V = g.V;
  const int *__restrict__ rp = g.csr_rp, *__restrict__ ci = g.csr_ci;
  const int lane = threadIdx.x & 31;
  const T* __restrict__ val = MIXED ? (const T*)a.val32 : (const T*)g.csr_val;
  const T* __restrict__ v = MIXED ? (const T*)a.pf : (const T*)a.p;
  T* __restrict__ q = MIXED ? (T*)a.qf : (T*)a.q;
  bool any = false;   // lanes whose slots all rest neither load nor store (an idle slot's q may be overwritten)
  T dot[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    any |= bk_on(a.st + lane * SPL + k, BK_AP);
    dot[k] = T(0);
  }
  const int tw = gridDim.x * (BT / 32);
  int i = blockIdx.x * (BT / 32) + (threadIdx.x >> 5);
  int b = 0, e = 0, b2 = 0, e2 = 0, c = 0;
  T w = T(0);
  if (i < V) {
    b = __ldg(rp + i);
    e = __ldg(rp + i + 1);
    if (i + tw < V) {
      b2 = __ldg(rp + i + tw);
      e2 = __ldg(rp + i + tw + 1);
    }
    if (b + lane < e) {
      c = __ldg(ci + b + lane);
      w = __ldg(val + b + lane);
    }
  }
  for (; i < V; i += tw) {
    int b3 = 0, e3 = 0, c2 = 0;
    T w2 = T(0);
    if (b2 + lane < e2) {
      c2 = __ldg(ci + b2 + lane);
      w2 = __ldg(val + b2 + lane);
    }
    if ((long long)i + 2LL * tw < V) {
      b3 = __ldg(rp + i + 2 * tw);
      e3 = __ldg(rp + i + 2 * tw + 1);
    }
    P own, acc;
#pragma unroll
    for (int k = 0; k < SPL; ++k) own.v[k] = acc.v[k] = T(0);
    if (any) own = *reinterpret_cast<const P*>(v + (size_t)i * B + lane * SPL);
    for (int e0 = b; e0 < e; e0 += 32) {
      const int n = min(32, e - e0);
      if (e0 != b) {   // a row of more than 32 entries
        c = lane < n ? __ldg(ci + e0 + lane) : 0;
        w = lane < n ? __ldg(val + e0 + lane) : T(0);
      }
      for (int j0 = 0; j0 < n; j0 += U) {
        P gv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int cj = __shfl_sync(FULL, c, j0 + u);
#pragma unroll
          for (int k = 0; k < SPL; ++k) gv[u].v[k] = T(0);
          if (any && j0 + u < n) gv[u] = *reinterpret_cast<const P*>(v + (size_t)cj * B + lane * SPL);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const T wj = __shfl_sync(FULL, w, j0 + u);   // lanes past the row hold 0
#pragma unroll
          for (int k = 0; k < SPL; ++k) acc.v[k] = fma(j0 + u < n ? wj : T(0), gv[u].v[k], acc.v[k]);
        }
      }
    }
    if (any) {
      *reinterpret_cast<P*>(q + (size_t)i * B + lane * SPL) = acc;
#pragma unroll
      for (int k = 0; k < SPL; ++k) dot[k] = fma(own.v[k], acc.v[k], dot[k]);
    }
    b = b2, e = e2, b2 = b3, e2 = e3, c = c2, w = w2;
  }
  bk_finish<B>(a, g, BK_AP, bk_sum_lanes<SPL>(dot));
}

// The streaming kernels: a thread owns VW neighbouring slots (16 bytes) of every (blocks BT / TPR)-th row and takes BR rows
// at a time, all loads first.  Slots at rest keep their values: a thread without a running slot skips its loads, the
// others write back what they read.
constexpr int BR = 2;
#define BK_STREAM(B, VW)                                                                                     \
  constexpr int TPR = (B) / (VW);                                                                            \
  const int slot0 = (int)(threadIdx.x % TPR) * (VW);                                                         \
  const int tw = (int)gridDim.x * (BT / TPR), row0 = (int)blockIdx.x * (BT / TPR) + (int)threadIdx.x / TPR;

// x += alpha p ; r -= alpha q ; (r, r)   (MIXED: the correction xl, r, p, q and the lane sums in FP32)
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(BT, 4) k_bcg_xr(BArgs a) {
  typedef typename std::conditional<MIXED, float, double>::type T;
  constexpr int B = 32 * SPL, VW = 16 / sizeof(T);
  typedef Pack<T, VW> P;
  const LatGeom& g = *a.lat;
  const int V = g.V;
  BK_STREAM(B, VW)
  bool on[VW], any = false;
  T al[VW], acc[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    const SlotState* S = a.st + slot0 + k;
    on[k] = bk_on(S, BK_XR);
    any |= on[k];
    al[k] = (T)S->alpha.x;
    acc[k] = T(0);
  }
  T* __restrict__ x = MIXED ? (T*)a.xl : (T*)a.x;
  T* __restrict__ r = MIXED ? (T*)a.rf : (T*)a.r;
  const T* __restrict__ p = MIXED ? (const T*)a.pf : (const T*)a.p;
  const T* __restrict__ q = MIXED ? (const T*)a.qf : (const T*)a.q;
  if (any)
    for (long long i0 = row0; i0 < V; i0 += (long long)BR * tw) {
      P xv[BR], pv[BR], qv[BR], rv[BR];
#pragma unroll
      for (int u = 0; u < BR; ++u) {
        const long long i = i0 + (long long)u * tw;
        if (i >= V) continue;
        const size_t o = (size_t)i * B + slot0;
        xv[u] = *reinterpret_cast<const P*>(x + o);
        pv[u] = *reinterpret_cast<const P*>(p + o);
        qv[u] = *reinterpret_cast<const P*>(q + o);
        rv[u] = *reinterpret_cast<const P*>(r + o);
      }
#pragma unroll
      for (int u = 0; u < BR; ++u) {
        const long long i = i0 + (long long)u * tw;
        if (i >= V) continue;
        const size_t o = (size_t)i * B + slot0;
#pragma unroll
        for (int k = 0; k < VW; ++k) {
          const T rn = fma(-al[k], qv[u].v[k], rv[u].v[k]), xn = fma(al[k], pv[u].v[k], xv[u].v[k]);
          if (on[k]) {
            xv[u].v[k] = xn;
            rv[u].v[k] = rn;
            acc[k] = fma(rn, rn, acc[k]);
          }
        }
        *reinterpret_cast<P*>(x + o) = xv[u];
        *reinterpret_cast<P*>(r + o) = rv[u];
      }
    }
  bk_finish<B>(a, g, BK_XR, bk_sum_cols<B, VW>(acc));
}

// p = r + beta p
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(BT, 4) k_bcg_p(BArgs a) {
  typedef typename std::conditional<MIXED, float, double>::type T;
  constexpr int B = 32 * SPL, VW = 16 / sizeof(T);
  typedef Pack<T, VW> P;
  const int V = a.lat->V;
  BK_STREAM(B, VW)
  bool on[VW], any = false;
  T be[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    const SlotState* S = a.st + slot0 + k;
    on[k] = S->status == SLOT_RUN;
    any |= on[k];
    be[k] = S->restart ? T(0) : (T)S->beta.x;
  }
  if (!any) return;
  T* __restrict__ p = MIXED ? (T*)a.pf : (T*)a.p;
  const T* __restrict__ r = MIXED ? (const T*)a.rf : (const T*)a.r;
  for (long long i0 = row0; i0 < V; i0 += (long long)BR * tw) {
    P pv[BR], rv[BR];
#pragma unroll
    for (int u = 0; u < BR; ++u) {
      const long long i = i0 + (long long)u * tw;
      if (i >= V) continue;
      pv[u] = *reinterpret_cast<const P*>(p + (size_t)i * B + slot0);
      rv[u] = *reinterpret_cast<const P*>(r + (size_t)i * B + slot0);
    }
#pragma unroll
    for (int u = 0; u < BR; ++u) {
      const long long i = i0 + (long long)u * tw;
      if (i >= V) continue;
#pragma unroll
      for (int k = 0; k < VW; ++k)
        if (on[k]) pv[u].v[k] = fma(be[k], pv[u].v[k], rv[u].v[k]);
      *reinterpret_cast<P*>(p + (size_t)i * B + slot0) = pv[u];
    }
  }
}

// q = b . x for the finished slots
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcg_quad(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  int m[SPL], pa[SPL];
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane * SPL + k;
    on[k] = bk_on(S, BK_QUAD);
    m[k] = S->m;
    pa[k] = S->a;
    acc[k] = 0.0;
  }
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k)
      if (on[k]) acc[k] += lap_source(g, i, m[k], pa[k]) * a.x[(size_t)i * B + lane * SPL + k];
  }
  bk_finish<B>(a, g, BK_QUAD, bk_sum_lanes<SPL>(acc));
}

// reliable update, first half (mixed precision: the matrix-vector product, the recurrences and the per-lane dot products
// run in FP32; ||b||^2, the block sums and the true residual b - A (xh + xl) in FP64): xh += xl, xl = 0 for the
// slots that asked for a true residual, which then recomputes r in FP64 and keeps p
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcm_fold(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  bool any = false;
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    on[k] = bk_on(a.st + lane * SPL + k, BK_TRUE);
    any |= on[k];
  }
  if (!__syncthreads_or(any)) return;
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      const size_t o = (size_t)i * B + lane * SPL + k;
      a.x[o] += (double)a.xl[o];
      a.xl[o] = 0.0f;
    }
  }
}

// True residual r = b - A x in FP64 for the slots that asked for one: most iterations none does, around an update several
// do.  The blocks list the asking slots (a slot is finalised by the last block that served it, so every block lists
// the same) and take them eight at a time, eight lanes per row (the entries are read once for eight slots, the gathers
// share sectors), or one at a time, one thread per row, where fewer than three ask.  MIXED: r is stored in FP32 for the
// iteration and the old p is kept.
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(256) k_btrue_slot(BArgs a, double* __restrict__ part, unsigned int* __restrict__ cnt) {
  constexpr int B = 32 * SPL;
  __shared__ int list[B], nask, last[8];
  __shared__ unsigned int words[SPL];
  __shared__ double sh[256];
  if (threadIdx.x < B) {
    const unsigned int w = __ballot_sync(0xffffffffu, a.st[threadIdx.x].need_update != 0);
    if ((threadIdx.x & 31) == 0) words[threadIdx.x >> 5] = w;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int n = 0;
    for (int k = 0; k < SPL; ++k)
      for (unsigned int w = words[k]; w; w &= w - 1) list[n++] = 32 * k + __ffs(w) - 1;
    nask = n;
  }
  __syncthreads();
  const int n = nask;
  if (n == 0) return;
  const LatGeom g = *a.lat;
  const int lsh = n >= 3 ? 3 : 0, L = 1 << lsh;
  const long long step = ((long long)gridDim.x * 256) >> lsh;
  for (int s0 = 0; s0 < n; s0 += L) {
    const int li = s0 + (int)(threadIdx.x & (L - 1));
    const int slot = li < n ? list[li] : -1;
    const int m = slot >= 0 ? a.st[slot].m : 0, pa = slot >= 0 ? a.st[slot].a : 0;
    double acc = 0.0;
    if (slot >= 0)
      for (long long i = ((long long)blockIdx.x * 256 + threadIdx.x) >> lsh; i < g.V; i += step) {
        double ax = 0.0;
        const int e1 = __ldg(g.csr_rp + i + 1);
        for (int e = __ldg(g.csr_rp + i); e < e1; ++e)
          ax += __ldg(g.csr_val + e) * a.x[(size_t)__ldg(g.csr_ci + e) * B + slot];
        const double rv = lap_source(g, (int)i, m, pa) - ax;
        if (MIXED)
          a.rf[(size_t)i * B + slot] = (float)rv;
        else
          a.r[(size_t)i * B + slot] = rv;
        acc += rv * rv;
      }
    __syncthreads();
    sh[threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {   // lane l adds the threads l, l + 32, ...: of its slot, since L divides 32
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) t += sh[threadIdx.x + 32 * w];
      for (int o = 16; o >= L; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (threadIdx.x < L && slot >= 0) {
        part[(size_t)slot * gridDim.x + blockIdx.x] = t;
        __threadfence();
        last[threadIdx.x] = atomicAdd(cnt + slot, 1u) == gridDim.x - 1u;
      } else if (threadIdx.x < 8) {
        last[threadIdx.x] = 0;
      }
    }
    __syncthreads();
    for (int l = 0; l < L; ++l) {
      if (!last[l]) continue;
      __threadfence();
      const int sl = list[s0 + l];
      double tot[1];
      block_sum_partials<1, 256>(part + (size_t)sl * gridDim.x, 0, gridDim.x, tot);
      if (threadIdx.x == 0) {
        cg_after_true(a.st + sl, tot[0], a.tol2, MIXED);
        cnt[sl] = 0;
      }
    }
  }
}

__global__ void k_to_f32(const double* __restrict__ in, long long n, float* __restrict__ out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = (float)in[i];
}

template <int SPL, bool MIXED>
struct BlockedSparseEngine {
  static constexpr int B = 32 * SPL;
  static constexpr int GROUP_MAX = B;   // the schedule's slot count is exactly B
  int kernels_per_iteration() const { return MIXED ? 5 : 4; }
  hp_ctx* ctx;
  BArgs a;
  int big_lat = 0;          // index of the largest lattice (set by the scheduler; unused here)
  bool one_lat = false;     // one lattice in the problem (set by the scheduler; unused here)
  int ntrue = 1;            // row blocks of the true-residual kernel (per slot)
  double* tpart = nullptr;  // its partial sums [B][ntrue]
  unsigned int* tcnt = nullptr;
  long long nnz = 0;
  double delta = 0.0;
  int group() const { return 1; }
  static constexpr bool MORE_SLOTS = false;   // rhs_block is always set
  hp_status setup(int ns, int Vmax, const LatGeom* lats_dev, SlotState* st, const hp_solver_opts& o, double tol,
                  double, const LatGeom&) {
    if (ns != B) {
      hp_set_error("blocked sparse CG: %d slots for a block of %d", ns, B);
      return HP_EINVAL;
    }
    memset(&a, 0, sizeof(a));
    a.lat = lats_dev;
    a.st = st;
    // one resident wave of the matrix-vector kernel (a second, partial wave would idle most SMs)
    int occ = 0;
    HP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)k_bcg_ap<SPL, MIXED>, BT, 0));
    const long long rows_blocks = ((long long)Vmax + BT / 32 - 1) / (BT / 32);   // one row per warp at least
    auto wave = [&](int blocks_per_sm) {
      return (int)std::max(1LL, std::min<long long>(rows_blocks, (long long)ctx->num_sms * std::max(blocks_per_sm, 1)));
    };
    a.nblk = wave(occ);
    a.nstream = wave(4);   // resident blocks of the streaming kernels
    const int nb = std::max(a.nblk, a.nstream);
    a.ngroups_max = (nb + 31) / 32;
    void* p = nullptr;
    ntrue = (int)std::max(1LL, std::min<long long>(((long long)Vmax + 255) / 256, (long long)ctx->num_sms * 8));
    HP_TRY(hp_ws(ctx, "bcg.tpart", sizeof(double) * (size_t)B * ntrue, &p));
    tpart = (double*)p;
    HP_TRY(hp_ws(ctx, "bcg.tcnt", sizeof(unsigned int) * B, &p));
    tcnt = (unsigned int*)p;
    HP_CUDA(cudaMemsetAsync(tcnt, 0, sizeof(unsigned int) * B, ctx->stream));
    HP_TRY(hp_ws(ctx, "bcg.part", sizeof(double) * (size_t)B * (nb + a.ngroups_max), &p));
    a.part = (double*)p;
    a.gpart = a.part + (size_t)B * nb;
    const size_t ncnt = sizeof(unsigned int) * BK_COUNT * (size_t)(1 + a.ngroups_max);
    HP_TRY(hp_ws(ctx, "bcg.cnt", ncnt, &p));
    a.cnt = (unsigned int*)p;
    HP_CUDA(cudaMemsetAsync(a.cnt, 0, ncnt, ctx->stream));
    const size_t fb = sizeof(double) * (size_t)B * Vmax;
    double** v[4] = {&a.x, &a.r, &a.p, &a.q};
    const char* names[4] = {"solve.lx", "solve.lr", "solve.lp", "solve.lq"};
    for (int k = 0; k < (MIXED ? 1 : 4); ++k) {
      HP_TRY(hp_ws(ctx, names[k], fb, &p));
      *v[k] = (double*)p;
      HP_CUDA(cudaMemsetAsync(p, 0, fb, ctx->stream));   // columns of idle slots stay finite
    }
    if (MIXED) {
      const size_t fs = sizeof(float) * (size_t)B * Vmax;
      float** vf[4] = {&a.xl, &a.rf, &a.pf, &a.qf};
      const char* nf[4] = {"solve.xl32", "solve.r32", "solve.p32", "solve.q32"};
      for (int k = 0; k < 4; ++k) {
        HP_TRY(hp_ws(ctx, nf[k], fs, &p));
        *vf[k] = (float*)p;
        HP_CUDA(cudaMemsetAsync(p, 0, fs, ctx->stream));
      }
      LatGeom g;   // the CSR values in FP32
      HP_CUDA(cudaMemcpyAsync(&g, lats_dev, sizeof(LatGeom), cudaMemcpyDeviceToHost, ctx->stream));
      HP_CUDA(cudaStreamSynchronize(ctx->stream));
      int e_end = 0;
      HP_CUDA(cudaMemcpyAsync(&e_end, g.csr_rp + g.V, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
      HP_CUDA(cudaStreamSynchronize(ctx->stream));
      nnz = e_end;
      HP_TRY(hp_ws(ctx, "bcg.val32", sizeof(float) * (size_t)std::max(nnz, 1LL), &p));
      a.val32 = (const float*)p;
      if (nnz) {
        ProfScope ps(ctx, "k_to_f32");
        k_to_f32<<<blocks_for(ctx, nnz, 256), 256, 0, ctx->stream>>>(g.csr_val, nnz, (float*)p);
      }
      HP_LAUNCH_CHECK();
      // default threshold: a true residual after every 10^5 reduction (measured on the renumbered
      // 64^3 grid: 1e-3 -> 4.0 updates per solve, 1e-4 -> 3.0, 1e-5 -> 2.1 with the FP64 iteration
      // count, 1e-6 -> 2.0 but 1.7% more iterations)
      const double d = o.delta > 0.0 ? o.delta : 1e-5;
      a.delta2 = d * d;
    }
    a.tol2 = tol * tol;
    a.maxiter = o.maxiter > 0 ? o.maxiter : 10000;
    return HP_OK;
  }
  hp_status init() {
    {
      ProfScope ps(ctx, MIXED ? "k_bcm_init" : "k_bcg_init");
      k_bcg_init<SPL, MIXED><<<a.nstream, BT, 0, ctx->stream>>>(a);
    }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
  hp_status iteration() {
    { ProfScope ps(ctx, MIXED ? "k_bcm_ap" : "k_bcg_ap"); k_bcg_ap<SPL, MIXED><<<a.nblk, BT, 0, ctx->stream>>>(a); }
    { ProfScope ps(ctx, MIXED ? "k_bcm_xr" : "k_bcg_xr"); k_bcg_xr<SPL, MIXED><<<a.nstream, BT, 0, ctx->stream>>>(a); }
    if (MIXED) {
      ProfScope ps(ctx, "k_bcm_fold");
      k_bcm_fold<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a);
    }
    {
      ProfScope ps(ctx, "k_btrue_slot");
      k_btrue_slot<SPL, MIXED><<<ntrue, 256, 0, ctx->stream>>>(a, tpart, tcnt);
    }
    { ProfScope ps(ctx, MIXED ? "k_bcm_p" : "k_bcg_p"); k_bcg_p<SPL, MIXED><<<a.nstream, BT, 0, ctx->stream>>>(a); }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
  hp_status keep(const std::vector<int>&, const std::vector<SlotState>&, const SolveProblem&) {
    hp_set_error("solutions are kept for the Wilson operator only");
    return HP_EUNSUPPORTED;
  }
  hp_status harvest(const std::vector<int>&, const SolveProblem&, int*) {
    { ProfScope ps(ctx, "k_bcg_quad"); k_bcg_quad<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
};

#include "hp_schedule.cuh"

// ------------------------------------------------------------------ one right-hand side per cluster
// A whole CG solve in one launch: a cluster of C thread blocks (C = 1, 2, 4, 8) owns one right-hand side, from the source to
// the quadrature.  The launches of the slot engine cost about 10 us each in dependent latencies (flags, block
// sums through L2, the scalar step), four of them an iteration, whatever the size; here a step ends in a cluster
// barrier, the block sums travel through distributed shared memory, and every block takes the scalar steps on its own
// copy of the state (the same sums in the same order, so all blocks agree on every branch and meet at every barrier).
// The vectors stay in global memory (L2), read with plain loads: other blocks of the cluster write them.
// Bound by the FP64 pipe (13 operations a site and iteration).
// 8^4, 256 vectors: 2746 -> 1472 us; 64^3, 32 vectors: 30.8 -> 24.0 ms.
__device__ __forceinline__ void cluster_barrier(int C) {
  if (C == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
}

template <int CLT>
struct ClusterSum {
  double sh[CLT];
  double in[2][8];   // the blocks' sums, two generations: a generation is read before the barrier after the next one's
};
// the cluster's sum of v in thread 0 of every block (other threads: undefined); a cluster barrier
template <int CLT>
__device__ __forceinline__ double cluster_sum(ClusterSum<CLT>& cs, double v, int C, int rank, int& gen) {
  cs.sh[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < CLT / 32; w += 2) t += cs.sh[threadIdx.x + 32 * w] + cs.sh[threadIdx.x + 32 * w + 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x < C) {
      const unsigned int mine = (unsigned int)__cvta_generic_to_shared(&cs.in[gen][rank]);
      unsigned int there;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(mine), "r"((unsigned int)threadIdx.x));
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(there), "d"(t) : "memory");
    }
  }
  cluster_barrier(C);
  double tot = 0.0;
  if (threadIdx.x == 0)
    for (int c = 0; c < C; ++c) tot += cs.in[gen][c];
  gen ^= 1;
  return tot;
}

template <bool MF, int CLT>
__device__ __forceinline__ void cg_cluster_solve(const LArgs& a, const LatGeom& g, SlotState& S, ClusterSum<CLT>& cs, int cid,
                                                 double* x, double* r, double* p, double* q, int C, int rank, int most) {
  const int lo = (int)((long long)g.V * rank / C), hi = (int)((long long)g.V * (rank + 1) / C);
  const int m = S.m, pa = S.a;
  const double diag0 = lap_diag0(g);
  int gen = 0;
  double acc = 0.0, tot;
  if (S.status == SLOT_INIT) {
    for (int i = lo + threadIdx.x; i < hi; i += CLT) {
      const double b = lap_src(g, a, cid, i, m, pa);
      x[i] = 0.0;
      r[i] = b;
      p[i] = b;
      acc = fma(b, b, acc);
    }
    tot = cluster_sum(cs, acc, C, rank, gen);
    if (threadIdx.x == 0) cg_after_init(&S, g, tot);
    __syncthreads();
  }
  // at most `most` iterations a launch; x, r, p and the state carry over to the next
  for (int it = 0; S.status == SLOT_RUN && it < most; ++it) {
    acc = 0.0;
    for (int i = lo + threadIdx.x; i < hi; i += 2 * CLT) {
      const int j = i + CLT;
      const double q0 = lap_site<MF, false>(g, diag0, p, i), q1 = j < hi ? lap_site<MF, false>(g, diag0, p, j) : 0.0;
      q[i] = q0;
      acc = fma(p[i], q0, acc);
      if (j < hi) {
        q[j] = q1;
        acc = fma(p[j], q1, acc);
      }
    }
    tot = cluster_sum(cs, acc, C, rank, gen);
    if (threadIdx.x == 0) cg_after_ap(&S, tot);
    __syncthreads();
    const double al = S.alpha.x;
    acc = 0.0;
    for (int i = lo + threadIdx.x; i < hi; i += 2 * CLT) {
      const int j = i + CLT < hi ? i + CLT : i;
      const double x0 = x[i], p0 = p[i], r0 = r[i], q0 = q[i], x1 = x[j], p1 = p[j], r1 = r[j], q1 = q[j];
      const double n0 = fma(-al, q0, r0), n1 = fma(-al, q1, r1);
      x[i] = fma(al, p0, x0);
      r[i] = n0;
      acc = fma(n0, n0, acc);
      if (j != i) {
        x[j] = fma(al, p1, x1);
        r[j] = n1;
        acc = fma(n1, n1, acc);
      }
    }
    tot = cluster_sum(cs, acc, C, rank, gen);
    if (threadIdx.x == 0) cg_after_xr(&S, g, tot, a.tol2, a.maxiter);
    __syncthreads();
    if (S.need_update) {   // the true residual r = b - A x
      acc = 0.0;
      for (int i = lo + threadIdx.x; i < hi; i += CLT) {
        const double rv = lap_src(g, a, cid, i, m, pa) - lap_site<MF, false>(g, diag0, x, i);
        r[i] = rv;
        acc = fma(rv, rv, acc);
      }
      tot = cluster_sum(cs, acc, C, rank, gen);
      if (threadIdx.x == 0) cg_after_true(&S, tot, a.tol2);
      __syncthreads();
    }
    if (S.status != SLOT_RUN) break;
    const double be = S.restart ? 0.0 : S.beta.x;
    for (int i = lo + threadIdx.x; i < hi; i += 2 * CLT) {
      const int j = i + CLT < hi ? i + CLT : i;
      const double p0 = p[i], r0 = r[i], p1 = p[j], r1 = r[j];
      p[i] = fma(be, p0, r0);
      if (j != i) p[j] = fma(be, p1, r1);
    }
    cluster_barrier(C);   // the next product reads the neighbours' p
  }
  if (S.status == SLOT_RUN) return;
  acc = 0.0;
  for (int i = lo + threadIdx.x; i < hi; i += CLT) acc = fma(lap_src(g, a, cid, i, m, pa), x[i], acc);
  tot = cluster_sum(cs, acc, C, rank, gen);   // no block leaves before the others have written their sums to it
  if (threadIdx.x == 0) S.q = make_double2(tot, 0.0);
}

// item = first + number of the cluster; the vectors of an item of the launch at its number times Vmax, its deflation
// coefficients at its number times defl_k.  (Vectors in
// shared memory, one block of 131 KB per SM, measured slower than two blocks with the vectors in L2: 8^4, 256 vectors 1.66
// against 1.47 ms.)
template <int CLT>
__global__ void __launch_bounds__(CLT, 1024 / CLT) k_cg_cluster(LArgs a, int first, int C, int most) {
  __shared__ SlotState S;
  __shared__ ClusterSum<CLT> cs;
  const int cid = blockIdx.x / C, rank = blockIdx.x - cid * C, item = first + cid;
  if (threadIdx.x == 0) S = a.st[item];
  __syncthreads();
  if (S.status != SLOT_INIT && S.status != SLOT_RUN) return;   // finished in an earlier launch (the whole cluster)
  const LatGeom g = a.lats[S.lat];
  const size_t off = (size_t)cid * a.Vmax;
  if (C > 1) cluster_barrier(C);   // every block of the cluster has started: its shared memory can be written
  if (g.mass_field) cg_cluster_solve<true, CLT>(a, g, S, cs, cid, a.x + off, a.r + off, a.p + off, a.q + off, C, rank, most);
  else cg_cluster_solve<false, CLT>(a, g, S, cs, cid, a.x + off, a.r + off, a.p + off, a.q + off, C, rank, most);
  __syncthreads();
  if (threadIdx.x == 0 && rank == 0) a.st[item] = S;
}

// How a problem of n right-hand sides of V sites (on average) runs: C blocks of `threads` per right-hand side, `wave`
// right-hand sides per launch; C = 0: the slot engine.
struct ClusterPlan {
  int C, threads, wave;
  int most;   // iterations per launch: about a second's worth at the most (a solve that needs more is launched again)
};
// The cost of an iteration over all right-hand sides in SM cycles: FP64 (6.5 cycles a site at 2 lanes per clock, at 0.8 of
// the rate; at half of it where a block is alone on its SM with more than L1 holds of its vectors) on the busiest SM
// plus the barriers, against the slot engine's FP64 over all SMs (0.7 of the rate) plus the latencies of its four
// launches.  At equal cost the larger cluster: two blocks of 512 threads share an SM and fill each other's waits; blocks
// that are alone on theirs take 1024 threads.  Both sides measured (clusters / slots): 64^3 with 32 vectors 24.0 / 30.8
// ms, 16 23.4 / 15.0, 64 58.5 / 60; 32^3 with 2 1.9 / 2.8, 64 5.6 / 8.0; 8^4 with 1 0.51 / 1.1, 64 0.55 / 1.75.
// Clusters of several blocks stop where they lose: 80^3 with 38 vectors 41.5 / 47.8 ms, 152 138 / 176; 96^3 with 38 95.6 /
// 76.5, 152 361 / 284; 128^3 with 38 184 / 175.  One block per right-hand side still wins there (96^3 with 304 vectors
// 402 / 564 ms), as far as the vectors of the resident blocks (two per SM) find room.
// A batch of uneven lattices takes at least as long as one solve of its largest on one cluster, against the slot engine's
// rounds of launches: 256 vectors of 8^4 with two of 64^3 took 53.7 ms with one block per right-hand side, 15.5 with four
// (slots 27); 64 of 8^4 with one of 64^3 13.7, slots 9.8.
// Room: 1 GB, else a 32nd of the device's memory (9.3 GB) and half of what is free or held for them already; the workspace
// stays with the context.
constexpr double CLUSTER_MAX_SITES = 600e3;   // of a cluster of several blocks
static hp_status cluster_plan(const hp_ctx* ctx, double n, double V, int Vmax, ClusterPlan* out) {
  ClusterPlan pl = {0, 512, 0, 0};
  const double per = 32.0 * Vmax, gb = (double)(1 << 30);   // four vectors
  double room = -1.0;
  const double slots = std::max(12.0, std::min(256.0, std::floor((double)(4 << 20) / Vmax)));
  const double rounds = Vmax > V ? std::ceil(n / slots) : 1.0;
  double best = 1.4 * n * V * 6.5 / ctx->num_sms + 60e3 * rounds;
  for (int C = 1; C <= 8; C *= 2) {
    if (C > 1 && (V < 1024.0 * C || Vmax > CLUSTER_MAX_SITES)) break;
    const double k = std::ceil(n * C / ctx->num_sms);   // blocks on the busiest SM
    const double alone = (Vmax / C > 8192.0 ? 1.9 : 1.25) * Vmax * 6.5 / C;
    const double cost = std::max(1.25 * k * V * 6.5 / C, alone) + (C == 1 ? 5e3 : 18e3);
    if (!(cost <= best)) continue;
    const double resident = std::min(n, std::max(1.0, (double)(2 * ctx->num_sms / C)));
    if (per * resident > gb) {
      if (room < 0.0) {
        size_t free_b = 0, total_b = 0, held = 0;
        HP_CUDA(cudaMemGetInfo(&free_b, &total_b));
        for (const char* name : {"solve.lx", "solve.lr", "solve.lp", "solve.lq"}) {
          auto it = ctx->ws.find(name);
          if (it != ctx->ws.end()) held += it->second.bytes;
        }
        room = std::min(total_b / 32.0, (free_b + held) / 2.0);
      }
      if (per * resident > room) continue;
    }
    best = cost;
    pl.C = C;
    pl.threads = k == 1.0 ? 1024 : 512;
    pl.wave = (int)std::min(n, std::max(resident, std::floor(gb / per)));
  }
  pl.most = (int)std::max(16.0, std::min(1024.0, 2e9 / best));
  *out = pl;
  return HP_OK;
}

static hp_status solve_laplace_clusters(hp_ctx* ctx, SolveProblem& pb, SolveResult& res, const ClusterPlan& pl) {
  const int C = pl.C, most = pl.most, wave = pl.wave;
  const auto t0 = std::chrono::steady_clock::now();
  const int nl = (int)pb.lats.size();
  int Vmax = 0;
  std::vector<SlotState> items;
  res.qj.assign(nl, {});
  res.qb.assign(nl, {});
  for (int L = 0; L < nl; ++L) {
    Vmax = std::max(Vmax, pb.lats[L].V);
    const int dof = pb.lats[L].parts;
    const size_t n = (size_t)(pb.s_max[L] - pb.first[L]) * dof;
    res.qj[L].assign(n, make_double2(0.0, 0.0));
    res.qb[L].assign(n, make_double2(0.0, 0.0));
    for (int64_t m = pb.first[L]; m < pb.s_max[L]; ++m)
      for (int k = 0; k < dof; ++k) {
        SlotState S;
        memset(&S, 0, sizeof(S));
        S.status = SLOT_INIT;
        S.lat = L;
        S.m = (int)m;
        S.a = k;
        items.push_back(S);
      }
  }
  const int n = (int)items.size();
  LArgs a;
  memset(&a, 0, sizeof(a));
  void* p = nullptr;
  HP_TRY(hp_ws(ctx, "solve.lats", sizeof(LatGeom) * nl, &p));
  HP_CUDA(cudaMemcpyAsync(p, pb.lats.data(), sizeof(LatGeom) * nl, cudaMemcpyHostToDevice, ctx->stream));
  a.lats = (const LatGeom*)p;
  HP_TRY(hp_ws(ctx, "solve.state", sizeof(SlotState) * (size_t)n, &p));
  a.st = (SlotState*)p;
  HP_CUDA(cudaMemcpyAsync(a.st, items.data(), sizeof(SlotState) * (size_t)n, cudaMemcpyHostToDevice, ctx->stream));
  a.Vmax = Vmax;
  a.nslots = wave;
  a.tol2 = pb.tol * pb.tol;
  a.maxiter = pb.opts.maxiter > 0 ? pb.opts.maxiter : 10000;
  const char* names[4] = {"solve.lx", "solve.lr", "solve.lp", "solve.lq"};
  double** v[4] = {&a.x, &a.r, &a.p, &a.q};
  for (int k = 0; k < 4; ++k) {
    HP_TRY(hp_ws(ctx, names[k], sizeof(double) * (size_t)wave * Vmax, &p));
    *v[k] = (double*)p;
  }
  const int defl_k = pb.lats[0].defl_k;
  if (defl_k) {
    HP_TRY(hp_ws(ctx, "solve.defl_c", sizeof(double) * (size_t)wave * defl_k, &p));
    a.dc = (double*)p;
  }
  int* dev_slots = nullptr;
  std::vector<int> ident;
  if (pb.want_grad) {
    HP_TRY(hp_ws(ctx, "solve.slots", sizeof(int) * (size_t)wave, &p));
    dev_slots = (int*)p;
    for (int i = 0; i < wave; ++i) ident.push_back(i);
    HP_CUDA(cudaMemcpyAsync(dev_slots, ident.data(), sizeof(int) * ident.size(), cudaMemcpyHostToDevice, ctx->stream));
  }
  void (*kern)(LArgs, int, int, int) = pl.threads == 1024 ? k_cg_cluster<1024> : k_cg_cluster<512>;
  for (int i0 = 0; i0 < n; i0 += wave) {
    const int nw = std::min(wave, n - i0);
    if (defl_k) {
      const int rows = 32768;   // grid limit of one dimension
      for (int j0 = 0; j0 < nw; j0 += rows) {
        LArgs b = a;
        b.st += i0 + j0;
        b.dc += (size_t)j0 * defl_k;
        ProfScope ps(ctx, "k_cg_defl");
        k_cg_defl<256><<<dim3(defl_k, std::min(rows, nw - j0)), 256, 0, ctx->stream>>>(b);
      }
      HP_LAUNCH_CHECK();
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(nw * C));
    cfg.blockDim = dim3(pl.threads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    for (bool again = true; again;) {
      {
        ProfScope ps(ctx, "k_cg_cluster");
        HP_CUDA(cudaLaunchKernelEx(&cfg, kern, a, i0, C, most));
      }
      again = false;
      if (a.maxiter > most) {
        HP_CUDA(cudaMemcpyAsync(items.data() + i0, a.st + i0, sizeof(SlotState) * (size_t)nw, cudaMemcpyDeviceToHost,
                                ctx->stream));
        HP_CUDA(cudaStreamSynchronize(ctx->stream));
        for (int i = i0; i < i0 + nw; ++i) again = again || items[i].status == SLOT_RUN;
      }
    }
    if (pb.want_grad) {
      LArgs b = a;
      b.st += i0;
      for (int L = 0; L < nl; ++L) {
        ProfScope ps(ctx, "k_lgrad");
        k_lgrad<<<lblocks(ctx, pb.lats[L].V, 256), 256, 0, ctx->stream>>>(b, L, dev_slots, nw, pb.grad_dev[L], pb.lats[L].V);
      }
      HP_LAUNCH_CHECK();
    }
  }
  HP_CUDA(cudaMemcpyAsync(items.data(), a.st, sizeof(SlotState) * (size_t)n, cudaMemcpyDeviceToHost, ctx->stream));
  HP_CUDA(cudaStreamSynchronize(ctx->stream));
  memset(&res.stats, 0, sizeof(res.stats));
  res.stats.iterations_min = 0x7fffffff;
  for (const SlotState& S : items) tally(S, pb.lats[S.lat].parts, pb, res);
  if (res.stats.rhs_solved == 0) res.stats.iterations_min = 0;
  res.stats.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  return HP_OK;
}

template <int SPL, bool MIXED>
static hp_status run_blocked(hp_ctx* ctx, SolveProblem& pb, SolveResult& res) {
  BlockedSparseEngine<SPL, MIXED> e{ctx};
  return run_schedule(ctx, e, pb, res, 12, 0.0);
}

hp_status hp_solve_laplace(hp_ctx* ctx, SolveProblem& pb, SolveResult& res) {
  if (pb.lats[0].csr_rp) {   // a general sparse matrix (always alone, without a gradient)
    // blocked engine: B slots (rhs_block rounded up to 32, 64 or 128).  Automatic, measured on the renumbered 64^3 grid:
    // 32 where the queue fits (16 right-hand sides 17.9 ms, 20.3 in a block of 64); 128 in FP32 where the queue fills
    // most of it (128 right-hand sides 50.5 ms, 61.2 in blocks of 64); else 64 (64 right-hand sides FP32 28.9 ms, 33.9
    // in a block of 128; FP64 64 ms, 95)
    const long long nq = (long long)(pb.s_max[0] - pb.first[0]) * pb.lats[0].parts;
    const bool mixed = pb.opts.precision == HP_PREC_MIXED_FP32;
    const bool automatic = pb.opts.rhs_block <= 0;
    const int want = automatic ? (nq <= 32 ? 32 : (mixed && nq > 96 ? 128 : 64)) : pb.opts.rhs_block;
    auto run = [&](int B) {
      pb.opts.rhs_block = B;
      if (mixed) return B == 32 ? run_blocked<1, true>(ctx, pb, res) : B == 64 ? run_blocked<2, true>(ctx, pb, res) : run_blocked<4, true>(ctx, pb, res);
      return B == 32 ? run_blocked<1, false>(ctx, pb, res) : B == 64 ? run_blocked<2, false>(ctx, pb, res) : run_blocked<4, false>(ctx, pb, res);
    };
    const hp_status st = run(want <= 32 ? 32 : (want <= 64 ? 64 : 128));
    if (st != HP_ENOMEM || !automatic || want <= 64) return st;
    HP_TRY(hp_ws_release(ctx, "solve."));   // a wide block that found no room (before its first launch)
    return run(64);
  }
  // the caller who fixes the slots, the chunk or the graph replay gets the slot engine
  if (pb.opts.rhs_block <= 0 && pb.opts.check_every <= 0 && !pb.opts.use_graph) {
    double n = 0.0, work = 0.0;
    int Vmax = 1;
    for (size_t L = 0; L < pb.lats.size(); ++L) {
      Vmax = std::max(Vmax, pb.lats[L].V);
      const double k = (double)(pb.s_max[L] - pb.first[L]) * pb.lats[L].parts;
      n += k;
      work += k * pb.lats[L].V;
    }
    ClusterPlan pl;
    HP_TRY(cluster_plan(ctx, n, work / n, Vmax, &pl));
    if (pl.C && n <= 1e6) {
      const hp_status st = solve_laplace_clusters(ctx, pb, res, pl);
      if (st != HP_ENOMEM) return st;
      HP_TRY(hp_ws_release(ctx, "solve."));   // no room for them (seen before the first launch): the slot engine takes less
    }
  }
  LaplaceEngine e{ctx};
  return run_schedule(ctx, e, pb, res, 12, 0.0);
}
