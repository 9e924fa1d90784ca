// Shifted periodic Laplacian (the control problem of Section 5):
//   (A x)(s) = (8 + m + mu(s)) x(s) - sum_mu [x(s + mu) + x(s - mu)]
// in FP64, and multi-right-hand-side CG for the quadratures v^H A^-1 v.
// A is real, so a complex probe is solved as two real right-hand sides
// (its real and imaginary parts); the cross terms of v^H x cancel because
// A is symmetric.
#include <algorithm>
#include <cmath>
#include <cstring>

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
// lanes per clock (8^4, 256 slots: see k_cg_xr).
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
  // keeps the scheduler at 4M sites' worth of slots: 128^2x64 with 32 vectors took 116 ms in 12 slots, 122 in 32
  static size_t slot_bytes(const LaplaceEngine&, int) { return (size_t)8 << 30; }
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
// [row][slot] (lane l of a warp owns slots l, l + 32, ...).  One warp per row reads the row's
// CSR entries once for every slot and gathers B contiguous values per entry (256 SPL bytes,
// whole sectors), where one slot per block row would re-read the matrix for every slot and
// gather single words.  Reductions: each block leaves per-slot partial sums, the last block
// to finish adds them in a fixed order and takes the scalar CG steps of every slot.
struct BArgs {
  const LatGeom* lat;
  SlotState* st;
  double *x, *r, *p, *q;   // [n][B]
  double* part;            // [B][nblk]
  unsigned int* cnt;       // one counter per reducing kernel
  int nblk;               // blocks of the matrix-vector kernels
  int nstream;            // blocks of the streaming kernels
  int pstride;            // row stride of part: max(nblk, nstream)
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

template <int SPL>
__device__ __forceinline__ void bk_finish(const BArgs& a, const LatGeom& g, int kind, const double (&acc)[SPL]) {
  constexpr int B = 32 * SPL, NW = BT / 32;
  __shared__ double sh[NW][B];
  __shared__ double tot_sh[B];
  __shared__ int am_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < SPL; ++k) sh[warp][lane + 32 * k] = acc[k];
  __syncthreads();
  if (threadIdx.x < B) {
    double t = 0.0;
    for (int w = 0; w < NW; ++w) t += sh[w][threadIdx.x];
    a.part[(size_t)threadIdx.x * a.pstride + blockIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = atomicAdd(a.cnt + kind, 1u) == (unsigned)gridDim.x - 1u;
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  // warp w adds up the partials of slots w, w + NW, ...: lanes run over the blocks (coalesced
  // loads, four independent sums each), then a shuffle tree; the order is fixed
  const int nb = gridDim.x;
  for (int s = warp; s < B; s += NW) {
    const double* ps = a.part + (size_t)s * a.pstride;
    double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
    int j = lane;
    for (; j + 96 < nb; j += 128) {
      t0 += __ldcg(ps + j);
      t1 += __ldcg(ps + j + 32);
      t2 += __ldcg(ps + j + 64);
      t3 += __ldcg(ps + j + 96);
    }
    for (; j < nb; j += 32) t0 += __ldcg(ps + j);
    double t = (t0 + t1) + (t2 + t3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) tot_sh[s] = t;
  }
  __syncthreads();
  if (threadIdx.x < B) {
    const double tot = tot_sh[threadIdx.x];
    SlotState* S = a.st + threadIdx.x;
    if (bk_on(S, kind)) {
      switch (kind) {
        case BK_INIT: cg_after_init(S, g, tot); break;
        case BK_AP: cg_after_ap(S, tot); break;
        case BK_XR: cg_after_xr(S, g, tot, a.tol2, a.maxiter, a.delta2); break;
        case BK_TRUE: cg_after_true(S, tot, a.tol2, a.xl != nullptr); break;
        default: S->q = make_double2(tot, 0.0); break;
      }
    }
  }
  if (threadIdx.x == 0) a.cnt[kind] = 0;
}

#define BK_ROWS(i) for (int i = blockIdx.x * (BT / 32) + (threadIdx.x >> 5); i < g.V; i += gridDim.x * (BT / 32))
// rows i0 + u tw, u < BR, per warp and step: a streaming kernel issues all their loads first
constexpr int BR = 4;
#define BK_ROW_BATCHES(i0, tw)                            \
  const int tw = gridDim.x * (BT / 32);                   \
  for (int i0 = blockIdx.x * (BT / 32) + (threadIdx.x >> 5); i0 < g.V; i0 += BR * tw)

// x = 0, r = p = b for the slots being filled; ||b||^2
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcg_init(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  int m[SPL], pa[SPL];
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = bk_on(S, BK_INIT);
    m[k] = S->m;
    pa[k] = S->a;
    acc[k] = 0.0;
  }
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      const size_t o = (size_t)i * B + lane + 32 * k;
      const double b = lap_source(g, i, m[k], pa[k]);
      a.x[o] = 0.0;
      a.r[o] = b;
      a.p[o] = b;
      acc[k] += b * b;
    }
  }
  bk_finish<SPL>(a, g, BK_INIT, acc);
}

// (A v)[i][slot] for the rows r0 .. r1-1 of one warp, handed to flush(i, value, own) row by row
// in order, with own = own_src[i][slot] (own_src may be NULL).  The rows'
// CSR entries are contiguous: the warp loads them 32 at a time (one entry per lane, coalesced;
// the next 32 are requested before the current ones are used), broadcasts each entry, and
// issues U gathers of B contiguous values before it adds them.  Each warp walks a long chain of
// dependent loads, so every load that can be issued early is.
template <int SPL, typename T, int U = 8, class Flush>
__device__ __forceinline__ void bk_spmv_rows(const LatGeom& g, const T* __restrict__ val, const T* __restrict__ v,
                                             const T* __restrict__ own_src, int r0, int r1, int lane,
                                             const bool (&on)[SPL], Flush&& flush) {
  constexpr int B = 32 * SPL;
  constexpr unsigned FULL = 0xffffffffu;
  if (r0 >= r1) return;
  int i = r0, rbase = r0;
  int rend_l = (rbase + lane < r1) ? __ldg(g.csr_rp + rbase + lane + 1) : 0x7fffffff;
  int row_end = __shfl_sync(FULL, rend_l, 0);
  T acc[SPL], own[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) acc[k] = T(0);
  auto advance = [&](int e) {   // flush every row that ends at entry e (empty rows included)
    while (i < r1 && row_end == e) {
#pragma unroll
      for (int k = 0; k < SPL; ++k) own[k] = (own_src && on[k]) ? own_src[(size_t)i * B + lane + 32 * k] : T(0);
      flush(i, acc, own);
#pragma unroll
      for (int k = 0; k < SPL; ++k) acc[k] = T(0);
      ++i;
      if (i - rbase == 32) {
        rbase = i;
        rend_l = (rbase + lane < r1) ? __ldg(g.csr_rp + rbase + lane + 1) : 0x7fffffff;
      }
      if (i < r1) row_end = __shfl_sync(FULL, rend_l, i - rbase);
    }
  };
  const int e_beg = __ldg(g.csr_rp + r0), e_fin = __ldg(g.csr_rp + r1);
  advance(e_beg);
  int c_n = e_beg + lane < e_fin ? __ldg(g.csr_ci + e_beg + lane) : 0;
  T w_n = e_beg + lane < e_fin ? __ldg(val + e_beg + lane) : T(0);
  for (int e0 = e_beg; e0 < e_fin; e0 += 32) {
    const int nb = min(32, e_fin - e0);
    const int c_l = c_n;
    const T w_l = w_n;
    const int en = e0 + 32 + lane;   // the next 32 entries, requested now
    c_n = en < e_fin ? __ldg(g.csr_ci + en) : 0;
    w_n = en < e_fin ? __ldg(val + en) : T(0);
    for (int j0 = 0; j0 < nb; j0 += U) {
      T gv[U][SPL];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int c = __shfl_sync(FULL, c_l, j0 + u);   // lanes past nb hold row 0: in bounds, unused
        const T* vj = v + (size_t)c * B + lane;
#pragma unroll
        for (int k = 0; k < SPL; ++k) gv[u][k] = (on[k] && j0 + u < nb) ? vj[32 * k] : T(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (j0 + u < nb) {
          const T w = __shfl_sync(FULL, w_l, j0 + u);
#pragma unroll
          for (int k = 0; k < SPL; ++k) acc[k] += w * gv[u][k];
          advance(e0 + j0 + u + 1);
        }
      }
    }
  }
}

// the contiguous rows of warp number gw of tw warps
__device__ __forceinline__ void bk_warp_rows(int n, int& r0, int& r1) {
  const int tw = gridDim.x * (BT / 32), gw = blockIdx.x * (BT / 32) + (threadIdx.x >> 5);
  const int chunk = (n + tw - 1) / tw;
  r0 = min(n, gw * chunk);
  r1 = min(n, r0 + chunk);
}

// q = A p ; (p, q)
template <int SPL>
__global__ void __launch_bounds__(BT, SPL == 1 ? 4 : (SPL == 2 ? 3 : 2)) k_bcg_ap(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    on[k] = bk_on(a.st + lane + 32 * k, BK_AP);
    acc[k] = 0.0;
  }
  int r0, r1;
  bk_warp_rows(g.V, r0, r1);
  bk_spmv_rows<SPL, double>(g, g.csr_val, a.p, a.p, r0, r1, lane, on, [&](int i, const double (&qv)[SPL], const double (&pv)[SPL]) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      a.q[(size_t)i * B + lane + 32 * k] = qv[k];
      acc[k] += pv[k] * qv[k];
    }
  });
  bk_finish<SPL>(a, g, BK_AP, acc);
}

// x += alpha p ; r -= alpha q ; (r, r)
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcg_xr(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  double al[SPL], acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = bk_on(S, BK_XR);
    al[k] = S->alpha.x;
    acc[k] = 0.0;
  }
  double* __restrict__ x = a.x;
  double* __restrict__ r = a.r;
  const double* __restrict__ p = a.p;
  const double* __restrict__ q = a.q;
  BK_ROW_BATCHES(i0, tw) {   // loads of BR rows first, then the updates: BR x 4 SPL loads in flight
    double xv[BR][SPL], pv[BR][SPL], qv[BR][SPL], rv[BR][SPL];
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        xv[u][k] = x[o];
        pv[u][k] = p[o];
        qv[u][k] = q[o];
        rv[u][k] = r[o];
      }
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        x[o] = xv[u][k] + al[k] * pv[u][k];
        const double rn = rv[u][k] - al[k] * qv[u][k];
        r[o] = rn;
        acc[k] += rn * rn;
      }
  }
  bk_finish<SPL>(a, g, BK_XR, acc);
}

// p = r + beta p
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcg_p(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  double be[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = S->status == SLOT_RUN;
    be[k] = S->restart ? 0.0 : S->beta.x;
  }
  double* __restrict__ p = a.p;
  const double* __restrict__ r = a.r;
  BK_ROW_BATCHES(i0, tw) {
    double pv[BR][SPL], rv[BR][SPL];
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        pv[u][k] = p[o];
        rv[u][k] = r[o];
      }
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        p[(size_t)i * B + lane + 32 * k] = rv[u][k] + be[k] * pv[u][k];
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
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = bk_on(S, BK_QUAD);
    m[k] = S->m;
    pa[k] = S->a;
    acc[k] = 0.0;
  }
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k)
      if (on[k]) acc[k] += lap_source(g, i, m[k], pa[k]) * a.x[(size_t)i * B + lane + 32 * k];
  }
  bk_finish<SPL>(a, g, BK_QUAD, acc);
}

// ---- mixed precision (FP32 iteration, FP64 reliable updates): the matrix-vector product,
// the recurrences and the per-lane dot products in FP32; ||b||^2, the block sums and the true
// residual b - A (xh + xl) in FP64.  A reliable update folds xl into xh, recomputes r in FP64
// and keeps p.

// xh = 0, xl = 0, r = p = b
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcm_init(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  int m[SPL], pa[SPL];
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = bk_on(S, BK_INIT);
    m[k] = S->m;
    pa[k] = S->a;
    acc[k] = 0.0;
  }
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      const size_t o = (size_t)i * B + lane + 32 * k;
      const double b = lap_source(g, i, m[k], pa[k]);
      a.x[o] = 0.0;
      a.xl[o] = 0.0f;
      a.rf[o] = (float)b;
      a.pf[o] = (float)b;
      acc[k] += b * b;
    }
  }
  bk_finish<SPL>(a, g, BK_INIT, acc);
}

// q = A p, (p, q) in FP32
template <int SPL>
__global__ void __launch_bounds__(BT, SPL <= 2 ? 4 : 2) k_bcm_ap(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  float accf[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    on[k] = bk_on(a.st + lane + 32 * k, BK_AP);
    accf[k] = 0.0f;
  }
  int r0, r1;
  bk_warp_rows(g.V, r0, r1);
  bk_spmv_rows<SPL, float, 16>(g, a.val32, a.pf, a.pf, r0, r1, lane, on,
                           [&](int i, const float (&qv)[SPL], const float (&pv)[SPL]) {
#pragma unroll
                             for (int k = 0; k < SPL; ++k) {
                               if (!on[k]) continue;
                               a.qf[(size_t)i * B + lane + 32 * k] = qv[k];
                               accf[k] = fmaf(pv[k], qv[k], accf[k]);
                             }
                           });
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) acc[k] = accf[k];
  bk_finish<SPL>(a, g, BK_AP, acc);
}

// xl += alpha p, r -= alpha q, (r, r) in FP32
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcm_xr(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  float al[SPL], accf[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = bk_on(S, BK_XR);
    al[k] = (float)S->alpha.x;
    accf[k] = 0.0f;
  }
  float* __restrict__ xl = a.xl;
  float* __restrict__ rf = a.rf;
  const float* __restrict__ pf = a.pf;
  const float* __restrict__ qf = a.qf;
  BK_ROW_BATCHES(i0, tw) {
    float xv[BR][SPL], pv[BR][SPL], qv[BR][SPL], rv[BR][SPL];
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        xv[u][k] = xl[o];
        pv[u][k] = pf[o];
        qv[u][k] = qf[o];
        rv[u][k] = rf[o];
      }
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        xl[o] = fmaf(al[k], pv[u][k], xv[u][k]);
        const float rn = fmaf(-al[k], qv[u][k], rv[u][k]);
        rf[o] = rn;
        accf[k] = fmaf(rn, rn, accf[k]);
      }
  }
  double acc[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) acc[k] = accf[k];
  bk_finish<SPL>(a, g, BK_XR, acc);
}

// reliable update, first half: xh += xl, xl = 0 for the slots that asked for a true residual
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcm_fold(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  bool any = false;
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    on[k] = bk_on(a.st + lane + 32 * k, BK_TRUE);
    any |= on[k];
  }
  if (!__syncthreads_or(any)) return;
  BK_ROWS(i) {
#pragma unroll
    for (int k = 0; k < SPL; ++k) {
      if (!on[k]) continue;
      const size_t o = (size_t)i * B + lane + 32 * k;
      a.x[o] += (double)a.xl[o];
      a.xl[o] = 0.0f;
    }
  }
}

// p = r + beta p in FP32
template <int SPL>
__global__ void __launch_bounds__(BT) k_bcm_p(BArgs a) {
  constexpr int B = 32 * SPL;
  const LatGeom g = *a.lat;
  const int lane = threadIdx.x & 31;
  bool on[SPL];
  float be[SPL];
#pragma unroll
  for (int k = 0; k < SPL; ++k) {
    const SlotState* S = a.st + lane + 32 * k;
    on[k] = S->status == SLOT_RUN;
    be[k] = S->restart ? 0.0f : (float)S->beta.x;
  }
  float* __restrict__ pf = a.pf;
  const float* __restrict__ rf = a.rf;
  BK_ROW_BATCHES(i0, tw) {
    float pv[BR][SPL], rv[BR][SPL];
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        const size_t o = (size_t)i * B + lane + 32 * k;
        pv[u][k] = pf[o];
        rv[u][k] = rf[o];
      }
#pragma unroll
    for (int u = 0; u < BR; ++u)
#pragma unroll
      for (int k = 0; k < SPL; ++k) {
        const int i = i0 + u * tw;
        if (i >= g.V || !on[k]) continue;
        pf[(size_t)i * B + lane + 32 * k] = fmaf(be[k], pv[u][k], rv[u][k]);
      }
  }
}

// True residual r = b - A x in FP64 for the slots that asked for one, one thread per row and a
// grid row per slot (most iterations one slot or none asks: a warp per row over all slots would
// walk the whole matrix for a single lane).  MIXED: r is stored in FP32 for the iteration and
// the old p is kept.
template <int SPL, bool MIXED>
__global__ void __launch_bounds__(256) k_btrue_slot(BArgs a, double* __restrict__ part, unsigned int* __restrict__ cnt) {
  constexpr int B = 32 * SPL;
  const int slot = blockIdx.y;
  SlotState* S = a.st + slot;
  if (!S->need_update) return;
  const LatGeom g = *a.lat;
  const int m = S->m, pa = S->a;
  double acc[1] = {0.0};
  for (int i = blockIdx.x * 256 + threadIdx.x; i < g.V; i += gridDim.x * 256) {
    double ax = 0.0;
    const int e1 = __ldg(g.csr_rp + i + 1);
    for (int e = __ldg(g.csr_rp + i); e < e1; ++e)
      ax += __ldg(g.csr_val + e) * a.x[(size_t)__ldg(g.csr_ci + e) * B + slot];
    const double rv = lap_source(g, i, m, pa) - ax;
    if (MIXED)
      a.rf[(size_t)i * B + slot] = (float)rv;
    else
      a.r[(size_t)i * B + slot] = rv;
    acc[0] += rv * rv;
  }
  lreduce<1, 256>(acc, part + (size_t)slot * gridDim.x, 0, blockIdx.x);
  if (last_block(cnt + slot, gridDim.x)) {
    double tot[1];
    block_sum_partials<1, 256>(part + (size_t)slot * gridDim.x, 0, gridDim.x, tot);
    if (threadIdx.x == 0) {
      cg_after_true(S, tot[0], a.tol2, MIXED);
      cnt[slot] = 0;
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
  static size_t slot_bytes(const BlockedSparseEngine&, int Vmax) { return 32 * (size_t)Vmax; }   // rhs_block is always set
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
    HP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, MIXED ? (const void*)k_bcm_ap<SPL>
                                                                       : (const void*)k_bcg_ap<SPL>, BT, 0));
    const long long rows_blocks = ((long long)Vmax + BT / 32 - 1) / (BT / 32);   // one row per warp at least
    auto wave = [&](int blocks_per_sm) {
      return (int)std::max(1LL, std::min<long long>(rows_blocks, (long long)ctx->num_sms * std::max(blocks_per_sm, 1)));
    };
    a.nblk = wave(occ);
    a.nstream = wave(2048 / BT);
    a.pstride = std::max(a.nblk, a.nstream);
    void* p = nullptr;
    ntrue = (int)std::max(1LL, std::min<long long>(((long long)Vmax + 255) / 256, (long long)ctx->num_sms * 2));
    HP_TRY(hp_ws(ctx, "bcg.tpart", sizeof(double) * (size_t)B * ntrue, &p));
    tpart = (double*)p;
    HP_TRY(hp_ws(ctx, "bcg.tcnt", sizeof(unsigned int) * B, &p));
    tcnt = (unsigned int*)p;
    HP_CUDA(cudaMemsetAsync(tcnt, 0, sizeof(unsigned int) * B, ctx->stream));
    HP_TRY(hp_ws(ctx, "bcg.part", sizeof(double) * (size_t)B * a.pstride, &p));
    a.part = (double*)p;
    HP_TRY(hp_ws(ctx, "bcg.cnt", sizeof(unsigned int) * BK_COUNT, &p));
    a.cnt = (unsigned int*)p;
    HP_CUDA(cudaMemsetAsync(a.cnt, 0, sizeof(unsigned int) * BK_COUNT, ctx->stream));
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
    if (MIXED) {
      ProfScope ps(ctx, "k_bcm_init");
      k_bcm_init<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a);
    } else {
      ProfScope ps(ctx, "k_bcg_init");
      k_bcg_init<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a);
    }
    HP_LAUNCH_CHECK();
    return HP_OK;
  }
  hp_status iteration() {
    if (MIXED) {
      { ProfScope ps(ctx, "k_bcm_ap"); k_bcm_ap<SPL><<<a.nblk, BT, 0, ctx->stream>>>(a); }
      { ProfScope ps(ctx, "k_bcm_xr"); k_bcm_xr<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
      { ProfScope ps(ctx, "k_bcm_fold"); k_bcm_fold<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
      {
        ProfScope ps(ctx, "k_btrue_slot");
        k_btrue_slot<SPL, true><<<dim3(ntrue, B), 256, 0, ctx->stream>>>(a, tpart, tcnt);
      }
      { ProfScope ps(ctx, "k_bcm_p"); k_bcm_p<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
      HP_LAUNCH_CHECK();
      return HP_OK;
    }
    { ProfScope ps(ctx, "k_bcg_ap"); k_bcg_ap<SPL><<<a.nblk, BT, 0, ctx->stream>>>(a); }
    { ProfScope ps(ctx, "k_bcg_xr"); k_bcg_xr<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
    {
      ProfScope ps(ctx, "k_btrue_slot");
      k_btrue_slot<SPL, false><<<dim3(ntrue, B), 256, 0, ctx->stream>>>(a, tpart, tcnt);
    }
    { ProfScope ps(ctx, "k_bcg_p"); k_bcg_p<SPL><<<a.nstream, BT, 0, ctx->stream>>>(a); }
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
__device__ __forceinline__ void cg_cluster_solve(const LArgs& a, const LatGeom& g, SlotState& S, ClusterSum<CLT>& cs, int item,
                                                 double* x, double* r, double* p, double* q, int C, int rank, int most) {
  const int lo = (int)((long long)g.V * rank / C), hi = (int)((long long)g.V * (rank + 1) / C);
  const int m = S.m, pa = S.a;
  const double diag0 = lap_diag0(g);
  int gen = 0;
  double acc = 0.0, tot;
  if (S.status == SLOT_INIT) {
    for (int i = lo + threadIdx.x; i < hi; i += CLT) {
      const double b = lap_src(g, a, item, i, m, pa);
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
        const double rv = lap_src(g, a, item, i, m, pa) - lap_site<MF, false>(g, diag0, x, i);
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
  for (int i = lo + threadIdx.x; i < hi; i += CLT) acc = fma(lap_src(g, a, item, i, m, pa), x[i], acc);
  tot = cluster_sum(cs, acc, C, rank, gen);   // no block leaves before the others have written their sums to it
  if (threadIdx.x == 0) S.q = make_double2(tot, 0.0);
}

// item = first + number of the cluster; the vectors of an item of the launch at its number times Vmax.  (Vectors in
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
  if (g.mass_field) cg_cluster_solve<true, CLT>(a, g, S, cs, item, a.x + off, a.r + off, a.p + off, a.q + off, C, rank, most);
  else cg_cluster_solve<false, CLT>(a, g, S, cs, item, a.x + off, a.r + off, a.p + off, a.q + off, C, rank, most);
  __syncthreads();
  if (threadIdx.x == 0 && rank == 0) a.st[item] = S;
}

// How a problem of n right-hand sides of V sites (on average) runs: C blocks of `threads` per right-hand side; C = 0: the
// slot engine.
struct ClusterPlan {
  int C, threads;
  int most;   // iterations per launch: about a second's worth at the most (a solve that needs more is launched again)
};
// The cost of an iteration over all right-hand sides in SM cycles: FP64 (6.5 cycles a site at 2 lanes per clock, at 0.8 of
// the rate; at half of it where a block is alone on its SM with more than L1 holds of its vectors) on the busiest SM
// plus the barriers, against the slot engine's FP64 over all SMs (0.7 of the rate) plus the latencies of its four
// launches.  At equal cost the larger cluster: two blocks of 512 threads share an SM and fill each other's waits; blocks
// that are alone on theirs take 1024 threads.  Both sides measured (clusters / slots): 64^3 with 32 vectors 24.0 / 30.8
// ms, 16 23.4 / 15.0, 64 58.5 / 60; 32^3 with 2 1.9 / 2.8, 64 5.6 / 8.0; 8^4 with 1 0.51 / 1.1, 64 0.55 / 1.75.
static ClusterPlan cluster_plan(const hp_ctx* ctx, double n, double V) {
  ClusterPlan pl = {0, 512, 0};
  double best = 1.4 * n * V * 6.5 / ctx->num_sms + 60e3;
  for (int C = 1; C <= 8; C *= 2) {
    if (C > 1 && V < 1024.0 * C) break;
    const double k = std::ceil(n * C / ctx->num_sms);   // blocks on the busiest SM
    const double cost = (k == 1.0 && V / C > 8192.0 ? 1.9 : 1.25 * k) * V * 6.5 / C + (C == 1 ? 5e3 : 18e3);
    if (cost <= best) {
      best = cost;
      pl.C = C;
      pl.threads = k == 1.0 ? 1024 : 512;
    }
  }
  pl.most = (int)std::max(16.0, std::min(1024.0, 2e9 / best));
  return pl;
}

static hp_status solve_laplace_clusters(hp_ctx* ctx, SolveProblem& pb, SolveResult& res, const ClusterPlan& pl) {
  const int C = pl.C, most = pl.most;
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
  // right-hand sides per launch: as many as are resident at once, up to 1 GB of vectors beyond that
  const int resident = std::max(1, 2 * ctx->num_sms / C);
  const int wave = (int)std::min<long long>(n, std::max<long long>(resident, (1LL << 30) / (32LL * Vmax)));
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
    HP_TRY(hp_ws(ctx, "solve.defl_c", sizeof(double) * (size_t)n * defl_k, &p));
    a.dc = (double*)p;
    const int rows = 32768;   // grid limit of one dimension
    for (int i0 = 0; i0 < n; i0 += rows) {
      LArgs b = a;
      b.st += i0;
      b.dc += (size_t)i0 * defl_k;
      ProfScope ps(ctx, "k_cg_defl");
      k_cg_defl<256><<<dim3(defl_k, std::min(rows, n - i0)), 256, 0, ctx->stream>>>(b);
    }
    HP_LAUNCH_CHECK();
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
    // blocked engine: B slots (rhs_block rounded up to 32, 64 or 128; automatic: 64, the fastest
    // on the renumbered 64^3 grid matrix in both precisions)
    const int want = pb.opts.rhs_block > 0 ? pb.opts.rhs_block : 64;
    const bool mixed = pb.opts.precision == HP_PREC_MIXED_FP32;
    pb.opts.rhs_block = want <= 32 ? 32 : (want <= 64 ? 64 : 128);
    if (mixed) {
      if (want <= 32) return run_blocked<1, true>(ctx, pb, res);
      if (want <= 64) return run_blocked<2, true>(ctx, pb, res);
      return run_blocked<4, true>(ctx, pb, res);
    }
    if (want <= 32) return run_blocked<1, false>(ctx, pb, res);
    if (want <= 64) return run_blocked<2, false>(ctx, pb, res);
    return run_blocked<4, false>(ctx, pb, res);
  }
  // the caller who fixes the slots, the chunk or the graph replay gets the slot engine
  if (pb.opts.rhs_block <= 0 && pb.opts.check_every <= 0 && !pb.opts.use_graph) {
    double n = 0.0, work = 0.0;
    for (size_t L = 0; L < pb.lats.size(); ++L) {
      const double k = (double)(pb.s_max[L] - pb.first[L]) * pb.lats[L].parts;
      n += k;
      work += k * pb.lats[L].V;
    }
    const ClusterPlan pl = cluster_plan(ctx, n, work / n);
    if (pl.C && n <= 1e6) return solve_laplace_clusters(ctx, pb, res, pl);
  }
  LaplaceEngine e{ctx};
  return run_schedule(ctx, e, pb, res, 12, 0.0);
}
