// Wilson-Dirac operator: link preparation and the dispatch of the apply, stencil benchmark and
// solver calls to the per-precision translation units (hp_wilson_impl.cuh: the stencil in
// FP64/FP32/FP16/BF16 and the multi-right-hand-side BiCGStab with FP64-class reliable updates
// that computes the quadratures v^H D^-1 v of the probing sources; Section 1.1.2: quadrature
// through a linear solve; Section 5.3: full spin-colour dilution).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>

#include "hp_fields.cuh"

// ============================================================ link preparation
// canonical complex128 [V][4][3][3]  ->  internal layouts
__global__ void k_links_convert(const double2* __restrict__ in, int V, double2* __restrict__ U64,
                                float4* __restrict__ U32, uint2* __restrict__ U16, float4* __restrict__ U32f,
                                float2* __restrict__ U32g, uint4* __restrict__ U16f, unsigned int* __restrict__ U16g,
                                float4* __restrict__ U32fl, float2* __restrict__ U32gl, int4* __restrict__ U32i,
                                int2* __restrict__ U32gi) {
  const long long total = 4LL * V;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int site = (int)(t >> 2), mu = (int)(t & 3);
    double2 u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = in[((size_t)site * 4 + mu) * 9 + k];
    if (U64) {
#pragma unroll
      for (int k = 0; k < 9; ++k) U64[((size_t)mu * 9 + k) * V + site] = u[k];
    }
    if (U32) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
        U32[((size_t)mu * 3 + k) * V + site] =
            make_float4((float)u[2 * k].x, (float)u[2 * k].y, (float)u[2 * k + 1].x, (float)u[2 * k + 1].y);
    }
    if (U16) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        uint2 v;
        v.x = Half2Ops<PR16>::from_f2((float)u[2 * k].x, (float)u[2 * k].y);
        v.y = Half2Ops<PR16>::from_f2((float)u[2 * k + 1].x, (float)u[2 * k + 1].y);
        U16[((size_t)mu * 3 + k) * V + site] = v;
      }
    }
    if (U32f) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        U32f[((size_t)mu * 4 + k) * V + site] =
            make_float4((float)u[2 * k].x, (float)u[2 * k].y, (float)u[2 * k + 1].x, (float)u[2 * k + 1].y);
      U32g[(size_t)mu * V + site] = make_float2((float)u[8].x, (float)u[8].y);
    }
    if (U32fl) {   // fixed-point links: 2^30 u = i + l, from the FP32 parts of u (u - (float)u is exact in FP32)
      int ii[18];
      float ll[18];
#pragma unroll
      for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const double v = c ? u[k].y : u[k].x;
          const float hi = (float)v, t = hi * 0x1p30f;
          const int a = __float2int_rn(t);
          const float r = fmaf((float)(v - (double)hi), 0x1p30f, t - (float)a);   // |r| <= 33
          const int b = __float2int_rn(r);
          ii[2 * k + c] = a + b;
          ll[2 * k + c] = r - (float)b;
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        U32i[((size_t)mu * 4 + k) * V + site] = make_int4(ii[4 * k], ii[4 * k + 1], ii[4 * k + 2], ii[4 * k + 3]);
        U32fl[((size_t)mu * 4 + k) * V + site] = make_float4(ll[4 * k], ll[4 * k + 1], ll[4 * k + 2], ll[4 * k + 3]);
      }
      U32gi[(size_t)mu * V + site] = make_int2(ii[16], ii[17]);
      U32gl[(size_t)mu * V + site] = make_float2(ll[16], ll[17]);
    }
    if (U16f) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint4 v;
        v.x = Half2Ops<PR16>::from_f2((float)u[4 * k].x, (float)u[4 * k].y);
        v.y = Half2Ops<PR16>::from_f2((float)u[4 * k + 1].x, (float)u[4 * k + 1].y);
        v.z = Half2Ops<PR16>::from_f2((float)u[4 * k + 2].x, (float)u[4 * k + 2].y);
        v.w = Half2Ops<PR16>::from_f2((float)u[4 * k + 3].x, (float)u[4 * k + 3].y);
        U16f[((size_t)mu * 2 + k) * V + site] = v;
      }
      U16g[(size_t)mu * V + site] = Half2Ops<PR16>::from_f2((float)u[8].x, (float)u[8].y);
    }
  }
}

__global__ void k_to_float(const double* __restrict__ in, float* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = (float)in[i];
}

hp_status hp_prepare_mass(hp_ctx* ctx, const hp_operator* op, LatGeom* g, const char* tag) {
  g->mass = op->mass;
  g->kappa = op->kappa;
  g->diag0 = (float)(1.0 + op->mass);
  g->mass_field = nullptr;
  g->mass_field32 = nullptr;
  if (op->mass_field) {
    std::string n = std::string(tag) + ".mass";
    const void* d = nullptr;
    HP_TRY(hp_device_view(ctx, op->mass_field, sizeof(double) * (size_t)g->V, n.c_str(), &d));
    g->mass_field = (const double*)d;
    void* f = nullptr;
    HP_TRY(hp_ws(ctx, (n + "32").c_str(), sizeof(float) * (size_t)g->V, &f));
    {
      ProfScope ps(ctx, "k_to_float");
      k_to_float<<<blocks_for(ctx, g->V, 256), 256, 0, ctx->stream>>>(g->mass_field, (float*)f, g->V);
    }
    HP_LAUNCH_CHECK();
    g->mass_field32 = (const float*)f;
  }
  return HP_OK;
}

// need_prec: bit mask of (1 << PR64) | (1 << PR32) | (1 << PR16)
hp_status hp_prepare_wilson(hp_ctx* ctx, const hp_operator* op, LatGeom* g, const char* tag, int need_prec) {
  if (!op->links) {
    hp_set_error("Wilson operator without links");
    return HP_EINVAL;
  }
  const size_t V = (size_t)g->V;
  std::string base(tag);
  const void* src = nullptr;
  // read once, by the conversion below: pinned host links stream in over the host link directly
  HP_TRY(hp_stream_view(ctx, op->links, sizeof(double) * 72 * V, (base + ".links_in").c_str(), &src));
  void *u64 = nullptr, *u32 = nullptr, *u16 = nullptr, *u32f = nullptr, *u32g = nullptr, *u16f = nullptr,
       *u16g = nullptr, *u32fl = nullptr, *u32gl = nullptr, *u32i = nullptr, *u32gi = nullptr;
  HP_TRY(hp_ws(ctx, (base + ".U64").c_str(), sizeof(double2) * 36 * V, &u64));   // always: true residual
  if (need_prec & (1 << PR32)) {
    HP_TRY(hp_ws(ctx, (base + ".U32").c_str(), sizeof(float4) * 12 * V, &u32));
    HP_TRY(hp_ws(ctx, (base + ".U32f").c_str(), sizeof(float4) * 16 * V, &u32f));
    HP_TRY(hp_ws(ctx, (base + ".U32g").c_str(), sizeof(float2) * 4 * V, &u32g));
    HP_TRY(hp_ws(ctx, (base + ".U32fl").c_str(), sizeof(float4) * 16 * V, &u32fl));
    HP_TRY(hp_ws(ctx, (base + ".U32gl").c_str(), sizeof(float2) * 4 * V, &u32gl));
    HP_TRY(hp_ws(ctx, (base + ".U32i").c_str(), sizeof(int4) * 16 * V, &u32i));
    HP_TRY(hp_ws(ctx, (base + ".U32gi").c_str(), sizeof(int2) * 4 * V, &u32gi));
  }
  if (need_prec & (1 << PR16)) {
    HP_TRY(hp_ws(ctx, (base + ".U16").c_str(), sizeof(uint2) * 12 * V, &u16));
    HP_TRY(hp_ws(ctx, (base + ".U16f").c_str(), sizeof(uint4) * 8 * V, &u16f));
    HP_TRY(hp_ws(ctx, (base + ".U16g").c_str(), sizeof(unsigned int) * 4 * V, &u16g));
  }
  {
    ProfScope ps(ctx, "k_links_convert");
    k_links_convert<<<blocks_for(ctx, 4LL * V, 256), 256, 0, ctx->stream>>>(
        (const double2*)src, (int)V, (double2*)u64, (float4*)u32, (uint2*)u16, (float4*)u32f, (float2*)u32g,
        (uint4*)u16f, (unsigned int*)u16g, (float4*)u32fl, (float2*)u32gl, (int4*)u32i, (int2*)u32gi);
  }
  HP_LAUNCH_CHECK();
  g->U64 = (const double2*)u64;
  g->U32 = (const float4*)u32;
  g->U16 = (const uint2*)u16;
  g->U32f = (const float4*)u32f;
  g->U32g = (const float2*)u32g;
  g->U16f = (const uint4*)u16f;
  g->U16g = (const unsigned int*)u16g;
  g->U32fl = (const float4*)u32fl;
  g->U32gl = (const float2*)u32gl;
  g->U32i = (const int4*)u32i;
  g->U32gi = (const int2*)u32gi;
  return hp_prepare_clover(ctx, op, g, tag);
}


// per-precision Wilson entry points (hp_wilson_<precision>.cu)
#define HP_WILSON_DECLARE(SUFFIX)                                                                             \
  hp_status hp_wilson_apply_##SUFFIX(hp_ctx* ctx, const LatGeom& g, int nrhs, const double* in, double* out); \
  hp_status hp_wilson_bench_##SUFFIX(hp_ctx* ctx, const LatGeom& g, int nrhs, int iters, double* ms);         \
  hp_status hp_wilson_schur_##SUFFIX(hp_ctx* ctx, const LatGeom& g, int nrhs, int eo_kernel, const double* in,   \
                                      double* out);                                                           \
  hp_status hp_wilson_solve_##SUFFIX(hp_ctx* ctx, SolveProblem& pb, SolveResult& res, bool eo, bool clover,   \
                                     double delta);
HP_WILSON_DECLARE(fp64)
HP_WILSON_DECLARE(fp32)
HP_WILSON_DECLARE(fp16)
HP_WILSON_DECLARE(bf16)

// ---- out = D in in FP64, straight from the canonical links and fields (no clover term)
// Bound by the FP64 pipe (2 lanes per clock and SM; 864 operations a site), so the fields need no other layout: the
// 16-byte loads of a site's 192 bytes meet in L1.  Two threads share a site: thread s computes spin s of the eight
// half spinors (projection, SU(3) product, its part of the reconstruction) and the output spins s and 2 + s; the lower
// partial sums that belong to the other thread change hands once.  Half the work per thread is what fills the GPU on
// a small lattice.  A link serves both threads of a site from one sector, and the blocks of one tile for all
// right-hand sides are launched next to each other, so links come from DRAM once.
// 8^4, one field: 21.7 us with five stream operations (links into every precision's layout, two layout passes, one
// thread per site) -> 8.7 us; 12 fields of 16^3x32: 2784 us -> 2481 us (2216 us at the FP64 rate).
template <int MU, int SIGN>
__device__ __forceinline__ void apply64_dir(const double2* __restrict__ psi, const double2* __restrict__ link, int s,
                                            double sg, double2 (&up)[3], double2 (&low)[3]) {
  // h = p_s + k p_t, k = +-i (directions 1, 3) or +-1 (2, 4); t = 3 - s (directions 1, 2) or 2 + s (3, 4)
  constexpr bool imag = MU == 0 || MU == 2;
  const double k = MU == 0 ? (SIGN < 0 ? 1.0 : -1.0) : MU == 3 ? (SIGN < 0 ? -1.0 : 1.0) : (SIGN < 0 ? sg : -sg);
  const double2* a = psi + 3 * s;
  const double2* b = psi + 3 * (MU < 2 ? 3 - s : 2 + s);
  double2 h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 x = __ldg(a + c), y = __ldg(b + c);
    h[c] = imag ? make_double2(fma(-k, y.y, x.x), fma(k, y.x, x.y)) : make_double2(fma(k, y.x, x.x), fma(k, y.y, x.y));
  }
  double2 u[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) u[e] = __ldg(link + e);
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    double wx = 0.0, wy = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 e = SIGN < 0 ? u[3 * r + c] : u[3 * c + r];
      const double ey = SIGN < 0 ? e.y : -e.y;   // U, or U^H for the backward neighbour
      wx = fma(e.x, h[c].x, wx);
      wx = fma(-ey, h[c].y, wx);
      wy = fma(e.x, h[c].y, wy);
      wy = fma(ey, h[c].x, wy);
    }
    up[r].x += wx;
    up[r].y += wy;
    // lower spin t += conj(k) w
    low[r] = imag ? make_double2(fma(k, wy, low[r].x), fma(-k, wx, low[r].y)) : make_double2(fma(k, wx, low[r].x), fma(k, wy, low[r].y));
  }
}

template <int NT>
__global__ void __launch_bounds__(NT) k_wilson_apply64(LatGeom g, const double2* __restrict__ links, const double2* __restrict__ in,
                                                       double2* __restrict__ out, int nrhs) {
  const int tile = blockIdx.x / nrhs, rhs = blockIdx.x - tile * nrhs;
  const long long t = (long long)tile * NT + threadIdx.x;
  const bool on = (t >> 1) < g.V;
  const int site = on ? (int)(t >> 1) : g.V - 1, s = (int)(t & 1);   // idle lanes repeat the last site: the exchange needs them
  int x[4], st[4];
  site_coords(g, site, x, st);
  const double2* f = in + (size_t)rhs * g.V * 12;
  const double sg = s == 0 ? 1.0 : -1.0;
  double2 up[3], la[3], lb[3];   // la: lower spin 3 - s (directions 1, 2); lb: lower spin 2 + s (directions 3, 4)
#pragma unroll
  for (int c = 0; c < 3; ++c) up[c] = la[c] = lb[c] = make_double2(0.0, 0.0);
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const int L = g.L[mu];
    const int fw = (x[mu] + 1 == L) ? site - (L - 1) * st[mu] : site + st[mu];
    const int bw = (x[mu] == 0) ? site + (L - 1) * st[mu] : site - st[mu];
    const double2 *pf = f + (size_t)fw * 12, *pb = f + (size_t)bw * 12;
    const double2 *uf = links + ((size_t)site * 4 + mu) * 9, *ub = links + ((size_t)bw * 4 + mu) * 9;
    if (mu == 0) { apply64_dir<0, -1>(pf, uf, s, sg, up, la); apply64_dir<0, 1>(pb, ub, s, sg, up, la); }
    if (mu == 1) { apply64_dir<1, -1>(pf, uf, s, sg, up, la); apply64_dir<1, 1>(pb, ub, s, sg, up, la); }
    if (mu == 2) { apply64_dir<2, -1>(pf, uf, s, sg, up, lb); apply64_dir<2, 1>(pb, ub, s, sg, up, lb); }
    if (mu == 3) { apply64_dir<3, -1>(pf, uf, s, sg, up, lb); apply64_dir<3, 1>(pb, ub, s, sg, up, lb); }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {   // the partner's la is this thread's lower spin 2 + s
    lb[c].x += __shfl_xor_sync(0xffffffffu, la[c].x, 1);
    lb[c].y += __shfl_xor_sync(0xffffffffu, la[c].y, 1);
  }
  if (!on) return;
  const double d = 1.0 + g.mass + (g.mass_field ? g.mass_field[site] : 0.0);
  const double2* c0 = f + (size_t)site * 12;
  double2* o = out + ((size_t)rhs * g.V + site) * 12;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 a = __ldg(c0 + 3 * s + c), b = __ldg(c0 + 6 + 3 * s + c);
    o[3 * s + c] = make_double2(fma(-g.kappa, up[c].x, d * a.x), fma(-g.kappa, up[c].y, d * a.y));
    o[6 + 3 * s + c] = make_double2(fma(-g.kappa, lb[c].x, d * b.x), fma(-g.kappa, lb[c].y, d * b.y));
  }
}

static bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return a && b && x < y + nb && y < x + na;
}

// the direct FP64 application; *done = false where it does not serve: an output that overlaps an input (threads write
// while others still read; the staged path copies every input first) or a grid beyond the launch limit
static hp_status apply_wilson_direct(hp_ctx* ctx, const hp_operator* op, LatGeom g, int nrhs, const double* in, double* out,
                                     bool* done) {
  const size_t V = (size_t)g.V, fb = sizeof(double2) * 12 * (size_t)nrhs * V, lb = sizeof(double) * 72 * V;
  const int NT = 2 * V * (size_t)nrhs >= (size_t)ctx->num_sms * 1024 ? 128 : 64;   // small: a block per SM before two
  const long long blocks = ((2 * (long long)V + NT - 1) / NT) * nrhs;
  *done = false;
  if (blocks > 0x7fffffffLL || overlap(out, fb, in, fb) || overlap(out, fb, op->links, lb) ||
      overlap(out, fb, op->mass_field, sizeof(double) * V))
    return HP_OK;
  const void *links = nullptr, *din = nullptr, *mf = nullptr;
  HP_TRY(hp_device_view(ctx, op->links, lb, "apply.links_in", &links));
  HP_TRY(hp_device_view(ctx, in, fb, "apply.canon_in", &din));
  g.mass = op->mass;
  g.kappa = op->kappa;
  if (op->mass_field) HP_TRY(hp_device_view(ctx, op->mass_field, sizeof(double) * V, "apply.mass", &mf));
  g.mass_field = (const double*)mf;
  double* dout = out;
  const bool out_host = !hp_is_device_ptr(out);
  if (out_host) {
    void* p = nullptr;
    HP_TRY(hp_ws(ctx, "apply.canon_out", fb, &p));
    dout = (double*)p;
  }
  {
    ProfScope ps(ctx, "k_wilson_apply64");
    if (NT == 64)
      k_wilson_apply64<64><<<(unsigned)blocks, 64, 0, ctx->stream>>>(g, (const double2*)links, (const double2*)din, (double2*)dout, nrhs);
    else
      k_wilson_apply64<128><<<(unsigned)blocks, 128, 0, ctx->stream>>>(g, (const double2*)links, (const double2*)din, (double2*)dout, nrhs);
  }
  HP_LAUNCH_CHECK();
  if (out_host) {
    HP_CUDA(cudaMemcpyAsync(out, dout, fb, cudaMemcpyDeviceToHost, ctx->stream));
    HP_CUDA(cudaStreamSynchronize(ctx->stream));
  }
  *done = true;
  return HP_OK;
}

hp_status hp_apply_wilson(hp_ctx* ctx, const hp_operator* op, LatGeom g, int nrhs, int prec, const double* in,
                          double* out) {
  if (prec == HP_PREC_FP64 && op->csw == 0.0) {
    bool done = false;
    HP_TRY(apply_wilson_direct(ctx, op, g, nrhs, in, out, &done));
    if (done) return HP_OK;
  }
  HP_TRY(hp_prepare_mass(ctx, op, &g, "apply"));
  // the link layouts of the precision asked for (the FP64 links are always made)
  const int need = prec == HP_PREC_FP64 ? 1 << PR64 : prec == HP_PREC_MIXED_FP32 ? 1 << PR32 : 1 << PR16;
  HP_TRY(hp_prepare_wilson(ctx, op, &g, "apply", need));
  switch (prec) {
    case HP_PREC_FP64: return hp_wilson_apply_fp64(ctx, g, nrhs, in, out);
    case HP_PREC_MIXED_FP32: return hp_wilson_apply_fp32(ctx, g, nrhs, in, out);
    case HP_PREC_MIXED_FP16: return hp_wilson_apply_fp16(ctx, g, nrhs, in, out);
    case HP_PREC_MIXED_BF16: return hp_wilson_apply_bf16(ctx, g, nrhs, in, out);
  }
  hp_set_error("unknown precision %d", prec);
  return HP_EINVAL;
}

// The red-black split behind the even-odd iteration: every hop must join sites of opposite parity,
// which holds when all four extents are even (an odd extent wraps around between sites of one
// parity; a padded extent 1 hops onto the site itself); the half-site numbering site >> 1 then
// needs L_1 even as well.
static bool eo_lattice(const LatGeom& g) {
  for (int j = 0; j < 4; ++j)
    if (g.L[j] % 2) return false;
  return true;
}

hp_status hp_schur_wilson(hp_ctx* ctx, const hp_operator* op, LatGeom g, int nrhs, int prec, int eo_kernel,
                          const double* in, double* out) {
  if (!eo_lattice(g)) {
    hp_set_error("the even-odd split needs every extent even (lattice %d x %d x %d x %d; an odd or a padded "
                 "extent joins sites of one parity)", g.L[0], g.L[1], g.L[2], g.L[3]);
    return HP_EINVAL;
  }
  if (op->kappa == 0.0) {
    hp_set_error("the Schur complement needs kappa != 0");
    return HP_EINVAL;
  }
  HP_TRY(hp_prepare_mass(ctx, op, &g, "schur"));
  HP_TRY(hp_prepare_wilson(ctx, op, &g, "schur", (1 << PR64) | (1 << PR32) | (1 << PR16)));
  switch (prec) {
    case HP_PREC_FP64: return hp_wilson_schur_fp64(ctx, g, nrhs, eo_kernel, in, out);
    case HP_PREC_MIXED_FP32: return hp_wilson_schur_fp32(ctx, g, nrhs, eo_kernel, in, out);
    case HP_PREC_MIXED_FP16: return hp_wilson_schur_fp16(ctx, g, nrhs, eo_kernel, in, out);
    case HP_PREC_MIXED_BF16: return hp_wilson_schur_bf16(ctx, g, nrhs, eo_kernel, in, out);
  }
  hp_set_error("unknown precision %d", prec);
  return HP_EINVAL;
}

hp_status hp_bench_wilson(hp_ctx* ctx, const hp_operator* op, LatGeom g, int prec, int nrhs, int iters, double* ms,
                          double* bytes, double* flops) {
  HP_TRY(hp_prepare_mass(ctx, op, &g, "bench"));
  HP_TRY(hp_prepare_wilson(ctx, op, &g, "bench", (1 << PR64) | (1 << PR32) | (1 << PR16)));
  double S = 0, L = 0;
  hp_status st = HP_EINVAL;
  switch (prec) {
    case HP_PREC_FP64: S = 192; L = 144; st = hp_wilson_bench_fp64(ctx, g, nrhs, iters, ms); break;
    case HP_PREC_MIXED_FP32: S = 96; L = 48; st = hp_wilson_bench_fp32(ctx, g, nrhs, iters, ms); break;
    case HP_PREC_MIXED_FP16: S = 52; L = 24; st = hp_wilson_bench_fp16(ctx, g, nrhs, iters, ms); break;
    case HP_PREC_MIXED_BF16: S = 52; L = 24; st = hp_wilson_bench_bf16(ctx, g, nrhs, iters, ms); break;
    default: hp_set_error("unknown precision %d", prec); return HP_EINVAL;
  }
  if (st != HP_OK) return st;
  *bytes = (double)nrhs * g.V * (2.0 * S + 4.0 * L / nrhs);
  *flops = 1368.0 * nrhs * g.V;
  return HP_OK;
}

hp_status hp_solve_wilson(hp_ctx* ctx, SolveProblem& pb, SolveResult& res) {
  const int prec = pb.opts.precision;
  double delta = pb.opts.delta;
  bool eo = pb.opts.even_odd != 0, clover = false;
  for (auto& g : pb.lats) {
    if (!eo_lattice(g)) eo = false;   // odd or padded extents: no red-black split, full-lattice iteration
    clover = clover || g.clover;
  }
  // default group-update thresholds per iteration precision (measured on the 32^3x64 workload)
  switch (prec) {
    case HP_PREC_FP64: return hp_wilson_solve_fp64(ctx, pb, res, eo, clover, delta > 0 ? delta : 0.0);
    case HP_PREC_MIXED_FP32: return hp_wilson_solve_fp32(ctx, pb, res, eo, clover, delta > 0 ? delta : 0.001);
    case HP_PREC_MIXED_FP16: return hp_wilson_solve_fp16(ctx, pb, res, eo, clover, delta > 0 ? delta : 0.03);
    case HP_PREC_MIXED_BF16: return hp_wilson_solve_bf16(ctx, pb, res, eo, clover, delta > 0 ? delta : 0.03);
  }
  hp_set_error("unknown precision %d", prec);
  return HP_EINVAL;
}
