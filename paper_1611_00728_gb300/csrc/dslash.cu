// Improved-staggered Dslash on CUDA cores (arXiv:1611.00728 Sec. 3: the
// generated "staggered dslash" kernel; Sec. 4: its least-data model bandwidth).
//
//   (D psi)(n) = sum_mu [ F_mu(n) psi(n+mu) - F_mu(n-mu)^+ psi(n-mu)
//                       + L_mu(n) psi(n+3mu) - L_mu(n-3mu)^+ psi(n-3mu) ]
//
// with eta_mu and the boundary sign already folded into F and L at load time.
// One thread computes one output site of one parity. Links are stored
// [parity][mu][elem][Vh] so that a warp reads each matrix element of 32
// consecutive sites as one contiguous segment; colour vectors are [3][Vh].
// The backward hop reads the forward link of the neighbour and applies the
// dagger in registers (forward-only storage, the standard MILC layout), or,
// with the 8-way option of the FP32 copy, reads -U^+ stored at the site itself.
// Neighbour indices are computed from the site coordinates (no index tables).
// With 12-real long links (FP32 copy only) the third row is rebuilt as
// conj(row0 x row1) / s, s = s0 * eta_mu * boundary sign of that link.
#include <math.h>

#include "dslash_core.cuh"
namespace {

using namespace dcore;

constexpr int kThreads = 128;

template <typename R, typename RO, bool RECON, bool EIGHT, int EPI>
__global__ void __launch_bounds__(kThreads, (sizeof(R) == 4 && EPI == EPI_SR_DOTS2) ? 9 : 0) k_dslash(DArgs<R> a) {
  typedef typename V2<R>::T R2;
  typedef typename V2<RO>::T O2;
  pdl_wait();
  pdl_launch_dependents();
  if (!gate_open(a.st, a.gate)) return;
  const int Vh = a.g.Vh;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double part = 0.0;
  float srs = 0.f, srq = 0.f, srr = 0.f;  // EPI_SR_DOTS*: the site's <r,s>, <r,q>, |r|^2 (FP32)
  float sdot = 0.f;                       // EPI_NORMAL_DOT with FP32 vectors: the site's dot
  if (i < Vh) {
    R2 acc[3];
    dslash_site<R, RECON, EIGHT>(a, i, acc);
    O2* out = static_cast<O2*>(a.out);
    if constexpr (EPI == EPI_PLAIN) {
#pragma unroll
      for (int c = 0; c < 3; ++c) out[(size_t)c * Vh + i] = mk<O2>((RO)acc[c].x, (RO)acc[c].y);
    } else if constexpr (EPI == EPI_NORMAL || EPI == EPI_NORMAL_DOT) {
      const R sig = (R)(a.sigma_dev ? *a.sigma_dev : a.sigma);
      const R2* yv = static_cast<const R2*>(a.y);
      R dot = R(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const R2 yc = ldg2(yv + (size_t)c * Vh + i);
        O2 o = mk<O2>((RO)(sig * yc.x - acc[c].x), (RO)(sig * yc.y - acc[c].y));
        out[(size_t)c * Vh + i] = o;
        dot = fma(yc.x, o.x, fma(yc.y, o.y, dot));
      }
      part = (double)dot;
      sdot = (float)dot;
    } else if constexpr (EPI == EPI_SR_DOTS || EPI == EPI_SR_DOTS2) {  // s = sigma r - D in; <r,s>, [<r,q>], |r|^2
      const R sig = (R)(a.sigma_dev ? *a.sigma_dev : a.sigma);
      const R2* rv = static_cast<const R2*>(a.y);
      const R2* qv = static_cast<const R2*>(a.y3);
      R rs = R(0), rq = R(0), rr = R(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const size_t k = (size_t)c * Vh + i;
        const R2 rc = ldg2(rv + k);
        O2 o = mk<O2>((RO)(sig * rc.x - acc[c].x), (RO)(sig * rc.y - acc[c].y));
        out[k] = o;
        rs = fma(rc.x, o.x, fma(rc.y, o.y, rs));
        rr = fma(rc.x, rc.x, fma(rc.y, rc.y, rr));
        if constexpr (EPI == EPI_SR_DOTS) {
          const R2 qc = ldg2(qv + k);
          rq = fma(rc.x, qc.x, fma(rc.y, qc.y, rq));
        }
      }
      srs = rs;
      srq = rq;
      srr = rr;
    } else {  // EPI_TRUE_RESID: out = b - sigma*x + D in, in FP64
      const double sig = a.sigma_dev ? *a.sigma_dev : a.sigma;
      const double2* xv = static_cast<const double2*>(a.y);
      O2* out2 = static_cast<O2*>(a.out2);
      double nrm = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double2 xc = __ldg(xv + (size_t)c * Vh + i);
        const double2 bc = __ldg(a.b + (size_t)c * Vh + i);
        const double re = bc.x - sig * xc.x + (double)acc[c].x;
        const double im = bc.y - sig * xc.y + (double)acc[c].y;
        O2 o = mk<O2>((RO)re, (RO)im);
        out[(size_t)c * Vh + i] = o;
        if (out2) out2[(size_t)c * Vh + i] = o;
        nrm += re * re + im * im;
      }
      part = nrm;
    }
  }
  if constexpr ((EPI == EPI_NORMAL_DOT && sizeof(R) == 8) || EPI == EPI_TRUE_RESID) {
    if (a.fin != FIN_NONE) block_partial(part, a.partials);
  } else if constexpr (EPI == EPI_NORMAL_DOT) {  // FP32: the site's dot is FP32; float-float partials
    if (a.fin != FIN_NONE) {
      float2 v[1] = {make_float2(sdot, 0.f)};
      block_sum_ffs<1>(v);
      if (threadIdx.x == 0) ffs_slots(a.partials)[blockIdx.x] = v[0];
    }
  }
  if constexpr (EPI == EPI_SR_DOTS) {  // float-float partials of the three sums
    if (a.fin != FIN_NONE) {
      float2 v[3] = {make_float2(srs, 0.f), make_float2(srq, 0.f), make_float2(srr, 0.f)};
      block_sum_ffs<3>(v);
      if (threadIdx.x == 0) {
        float2* slot = ffs_slots(a.partials);
        slot[blockIdx.x] = v[0];
        slot[gridDim.x + blockIdx.x] = v[1];
        slot[2 * gridDim.x + blockIdx.x] = v[2];
      }
    }
  } else if constexpr (EPI == EPI_SR_DOTS2) {  // sums 1 and 3 (the second comes from the update kernel)
    if (a.fin != FIN_NONE) {
      float2 v[2] = {make_float2(srs, 0.f), make_float2(srr, 0.f)};
      block_sum_ffs<2>(v);
      if (threadIdx.x == 0) {
        float2* slot = ffs_slots(a.partials);
        slot[blockIdx.x] = v[0];
        slot[2 * gridDim.x + blockIdx.x] = v[1];
      }
    }
  }
  (void)srs; (void)srq; (void)srr; (void)sdot;
}

// The same passes with a site's hops split over warps (dslash_split() says where): a block takes 32
// consecutive output sites; of its SPLIT warps, warp w does 16 / SPLIT of their hops (dslash_part), the
// partial sums meet in shared memory and warp c < 3 runs the epilogue of colour c.
//
// What bounds the one-thread form on a small lattice is the chain of 16 hops in a thread, each waiting for
// its loads: at 8^4 there are 16 blocks on 152 SMs and a pass takes 7.7 us (FP32, full links) whatever the
// rest of the chip does. Split, the chain is two hops and eight times the warps are in flight: 2.5 us
// (FP64 22.8 -> 7.3 us; timed in a graph of 20 launches, links in L2). The gate of a captured loop is read
// while the hops run and decides at the barrier: a block lives for about two loads, and waiting for the
// state first would add a third.
template <typename R, bool RECON, bool EIGHT, int SPLIT>
__global__ void __launch_bounds__(32 * SPLIT) k_dslash_split(DArgs<R> a) {
  typedef typename V2<R>::T R2;
  __shared__ R2 sm[SPLIT][3][32];
  __shared__ int open;
  pdl_wait();
  pdl_launch_dependents();
  const bool first = threadIdx.x == 0 && threadIdx.y == 0;
  const GateWords gw = gate_load(a.st, a.gate, first);
  const int Vh = a.g.Vh;
  const int i = blockIdx.x * 32 + threadIdx.x, c = threadIdx.y;
  const bool valid = i < Vh;
  if (valid) {
    R2 acc[3];
    dslash_part<R, RECON, EIGHT, SPLIT>(a, i, threadIdx.y, acc, PlainIn<R2, true>{a.in, Vh});
#pragma unroll
    for (int k = 0; k < 3; ++k) sm[threadIdx.y][k][threadIdx.x] = acc[k];
  }
  if (first) open = gate_value(gw, a.gate);
  __syncthreads();
  if (!open) return;
  double part = 0.0;                 // FP64 arithmetic: the colour's dot or norm
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;  // FP32: the colour's <y, out>, <y, q>, |y|^2
  if (c < 3 && valid) {
    R2 d = sm[0][c][threadIdx.x];
#pragma unroll
    for (int w = 1; w < SPLIT; ++w) {
      const R2 u = sm[w][c][threadIdx.x];
      d.x += u.x;
      d.y += u.y;
    }
    const size_t k = (size_t)c * Vh + i;
    if (a.epi == EPI_PLAIN) {
      static_cast<R2*>(a.out)[k] = d;
    } else if (a.epi == EPI_TRUE_RESID) {  // b - sigma x + D in, in FP64
      const double sig = a.sigma_dev ? *a.sigma_dev : a.sigma;
      const double2 xc = __ldg(static_cast<const double2*>(a.y) + k);
      const double2 bc = __ldg(a.b + k);
      const double re = bc.x - sig * xc.x + (double)d.x, im = bc.y - sig * xc.y + (double)d.y;
      if (a.out_f32) {
        const float2 o = make_float2((float)re, (float)im);
        static_cast<float2*>(a.out)[k] = o;
        if (a.out2) static_cast<float2*>(a.out2)[k] = o;
      } else {
        const double2 o = make_double2(re, im);
        static_cast<double2*>(a.out)[k] = o;
        if (a.out2) static_cast<double2*>(a.out2)[k] = o;
      }
      part = re * re + im * im;
    } else {  // sigma y - D in, and its sums
      const R sig = (R)(a.sigma_dev ? *a.sigma_dev : a.sigma);
      const R2 yc = ldg2(static_cast<const R2*>(a.y) + k);
      const R2 o = mk<R2>(sig * yc.x - d.x, sig * yc.y - d.y);
      static_cast<R2*>(a.out)[k] = o;
      const R dot = fma(yc.x, o.x, yc.y * o.y);
      part = (double)dot;
      s0 = (float)dot;
      if (a.epi == EPI_SR_DOTS || a.epi == EPI_SR_DOTS2) s2 = (float)fma(yc.x, yc.x, yc.y * yc.y);
      if (a.epi == EPI_SR_DOTS) {
        const R2 qc = ldg2(static_cast<const R2*>(a.y3) + k);
        s1 = (float)fma(yc.x, qc.x, yc.y * qc.y);
      }
    }
  }
  if (a.fin == FIN_NONE || a.epi == EPI_PLAIN || a.epi == EPI_NORMAL) return;
  if (sizeof(R) == 8) {
    const double t = colour_sum(part);
    if (first) a.partials[blockIdx.x] = t;
  } else {
    float2 v[3] = {make_float2(s0, 0.f), make_float2(s1, 0.f), make_float2(s2, 0.f)};
    colour_sum_ffs<3>(v);
    if (first) {
      float2* slot = ffs_slots(a.partials);
      slot[blockIdx.x] = v[0];
      if (a.epi == EPI_SR_DOTS) slot[gridDim.x + blockIdx.x] = v[1];
      if (a.epi != EPI_NORMAL_DOT) slot[2 * gridDim.x + blockIdx.x] = v[2];
    }
  }
}

template <typename R, typename RO, bool RECON, bool EIGHT>
int launch_t(sqcg_ctx* ctx, const DslashLaunch& L, cudaStream_t s) {
  typedef typename V2<R>::T R2;
  DArgs<R> a;
  a.g = ctx->g;
  a.par = L.out_parity;
  const int p = L.out_parity, q = 1 - L.out_parity;
  const size_t Vh = ctx->g.Vh;
  const int nl = RECON ? 6 : 9;  // the 12-real form exists for the FP32 copy only
  const R2* fat = reinterpret_cast<const R2*>(L.prec == SQCG_F64 ? (const void*)ctx->fat64 : (const void*)ctx->fat32);
  const R2* lng = reinterpret_cast<const R2*>(L.prec == SQCG_F64 ? (const void*)ctx->lng64 : (const void*)ctx->lng32);
  a.fat_p = fat + (size_t)p * 4 * 9 * Vh;
  a.fat_q = fat + (size_t)q * 4 * 9 * Vh;
  a.lng_p = lng + (size_t)p * 4 * nl * Vh;
  a.lng_q = lng + (size_t)q * 4 * nl * Vh;
  a.fatb_p = EIGHT ? reinterpret_cast<const R2*>(ctx->fatb32) + (size_t)p * 4 * 9 * Vh : nullptr;
  a.lngb_p = EIGHT ? reinterpret_cast<const R2*>(ctx->lngb32) + (size_t)p * 4 * nl * Vh : nullptr;
  a.nl = nl;
  a.inv_s0 = (R)(RECON ? 1.0 / ctx->long_scale : 1.0);
  a.in = static_cast<const R2*>(L.in);
  a.out = L.out;
  a.out2 = L.out2;
  a.y = L.y;
  a.y3 = L.y3;
  a.b = static_cast<const double2*>(L.b);
  a.sigma = L.sigma;
  a.sigma_dev = L.sigma_dev;
  a.st = ctx->st;
  a.partials = ctx->partials;
  a.gate = L.gate;
  a.fin = L.fin;
  if ((L.gate != GATE_NONE || L.fin != FIN_NONE) && (ctx->st == nullptr || ctx->partials == nullptr))
    return SQCG_ERR_INVALID_ARG;
  a.epi = L.epi;
  a.out_f32 = sizeof(RO) == 4;
  const bool sr = L.epi == EPI_SR_DOTS || L.epi == EPI_SR_DOTS2;
  const bool reduces = (L.epi == EPI_NORMAL_DOT || sr || L.epi == EPI_TRUE_RESID) && L.fin != FIN_NONE;
  const int split = dslash_split(ctx, L.prec, L.gate != GATE_NONE, L.pair != 0);
  const int grid = grid_for(ctx->g.Vh, split > 1 ? 32 : kThreads);
  if (reduces && grid > ctx->max_blocks) return SQCG_ERR_INVALID_ARG;  // partials hold 3 sums and more
  // programmatic dependent launch where the caller says a kernel precedes this one, and for the
  // finisher, which always follows the Dslash
  const bool pdl = L.pdl && ctx->pdl, fpdl = ctx->pdl != 0;
  void (*kern)(DArgs<R>) = nullptr;
  switch (L.epi) {
    case EPI_PLAIN: kern = k_dslash<R, RO, RECON, EIGHT, EPI_PLAIN>; break;
    case EPI_NORMAL: kern = k_dslash<R, RO, RECON, EIGHT, EPI_NORMAL>; break;
    case EPI_NORMAL_DOT: kern = k_dslash<R, RO, RECON, EIGHT, EPI_NORMAL_DOT>; break;
    case EPI_TRUE_RESID: kern = k_dslash<R, RO, RECON, EIGHT, EPI_TRUE_RESID>; break;
    case EPI_SR_DOTS: kern = k_dslash<R, RO, RECON, EIGHT, EPI_SR_DOTS>; break;
    case EPI_SR_DOTS2: kern = k_dslash<R, RO, RECON, EIGHT, EPI_SR_DOTS2>; break;
    default: return SQCG_ERR_INVALID_ARG;
  }
  dim3 block(kThreads);
  if (split > 1) {
    block = dim3(32, split);
    kern = split == 4 ? k_dslash_split<R, RECON, EIGHT, 4> : k_dslash_split<R, RECON, EIGHT, 8>;
  }
  SQCG_CUDA_TRY(launch_kernel(kern, grid, block, 0, s, pdl, a));
  if (reduces)
    return L.epi == EPI_SR_DOTS ? launch_finish_sr(ctx, grid, grid, grid, L.gate, s, fpdl)
           : L.epi == EPI_SR_DOTS2
               ? launch_finish_sr(ctx, grid, sr_update_partials(ctx), blas_grid(ctx), L.gate, s, fpdl)
           : (L.epi == EPI_NORMAL_DOT && sizeof(R) == 4) ? launch_finish_ffs(ctx, grid, L.fin, L.gate, s, fpdl)
                                                          : launch_finish(ctx, grid, L.fin, L.gate, s, fpdl);
  return SQCG_OK;
}

template <typename R, typename RO>
int launch_r(sqcg_ctx* ctx, const DslashLaunch& L, cudaStream_t s) {
  if constexpr (sizeof(R) == 4) {  // 12-real and 8-way forms exist for the FP32 copy only
    if (ctx->eightway)
      return ctx->recon ? launch_t<R, RO, true, true>(ctx, L, s) : launch_t<R, RO, false, true>(ctx, L, s);
    if (ctx->recon) return launch_t<R, RO, true, false>(ctx, L, s);
  }
  return launch_t<R, RO, false, false>(ctx, L, s);
}

}  // namespace

// By t, the 128-site tiles a SM. Two things decide: the chain of a site's 16 hops, which the split shortens where a SM
// has few warps, and how full the last wave is. One thread a site: 10 blocks of 128 a SM are resident (FP32, full
// links; 9 with 12-real ones, 8 with 8-way 12-real ones and in float-float), and a wave that ends just full beats the
// split, which does more work a site; one that starts anew loses to it. FP64 is bound by its pipe: a tile a SM
// takes 20 us, whole tiles with one thread a site, 32-site groups (of 5.4) with four warps.
// Measured on the GB300 (us a call, back to back; 1 / 4 / 8 warps a site group; loops: us of a whole solve):
//   FP32 full      Dslash   8^4 [t 0.1] 10.3/6.0/4.5, 16^4 [1.7] 10.3/6.3/8.2, 20^4 [4.1] 16.9/15.5/14.5, 22^4 [6.0]
//                           30.8/30.8/26.8, 24^4 [8.5] 35.0/39.0/35.0, 22x24x26x28 [9.9] 38.9/42.9/40.8, 26^4 [11.8]
//                           57.5/50.9/45.8, 32^4 [27] 98.5/104/94.9
//                  normal   18x20^3 [3.7] 28.8/28.6/27.1, 16x24x28x30 [8.3] 69.6/77.8/70.4, 24^4 70.0/79.8/73.3,
//                           20x20x28x32 [9.2] 74.0/82.7/78.1, 16x24x32x32 [10.1] 109/92/83
//                  8-way    normal 18x22x24x32 [7.8] 69.8/72.2/68.6, 24^4 72.1/75.9/73.3, 20x20x28x32 74.6/79.8/78.2
//                  CG loop  20x20x22x22 [5.0] 12797/12809/12656, 22^4 14591/16688/15314; multi-shift, 4 shifts, 16^3x32
//                           26246/23711/21970
//   FP32 12-real   Dslash   8^4 6.3/4.7/4.6, 14^4 [1.0] 8.2/6.0/6.1, 16^4 8.3/6.3/8.3, 14^2x24^2 8.3/10.3/10.4, 32^4
//                           81.8/83/83
//                  8-way    Dslash 12x14x24x24 [2.5] 8.3/8.3/10.3, 18^4 8.3/10.3/10.3, 18x22x24x32 26.0/30.8/29.2, 16x22x28x32
//                           [8.1] 34.9/30.8/30.8, 20x20x28x32 35.5/35.0/33.7; normal (both parities' links, past L2
//                           sooner) 18^4 29.0/26.8/25.5, 18x20x20x24 [4.4] 37.6/37.0/39.8, 20^3x22 [4.5] 37.5/42.5/39.4,
//                           24^4 63.6/64.7/66.6
//   FP64           Dslash   8^4 22.8/8.5/7.3, 14^4 24.7/22.7/24.7, 16^4 39.1/37.0/39.1, 12x18x18x20 [2.0] 41.1/43.2/45.2,
//                           14^2x24^2 59.6/63.7/65.7, 18x20^3 80.1/78.0/80.2, 16x18x18x30 [4.0] 80.1/82.4/86.1, 22^4
//                           133.5/124.9/129.3, 24^4 172/171/179; CG loop 16^4 14893/15286/14206, 12x16x16x22 [1.74]
//                           16989/17517/16223, 12x14x20x22 [1.9] 17383/19364/18707
//   float-float    Dslash   8^4 14.4/5.1/3.8, 16^4 16.6/14.4/14.5, 20x20x22x22 46.7/43.4/45.2, 18x20x22x26 [5.3] 48.4/
//                           51.3/51.1, 18x22x24x32 60.1/67.6/69.3, 16x22x28x32 86.3/68.2/72.6, 24x24x24x32 [11.4] 95/93/98
int dslash_split(const sqcg_ctx* ctx, int prec, bool loop, bool pair) {
  const double t = (double)grid_for(ctx->g.Vh, kThreads) / ctx->nsm;
  if (prec == SQCG_F32 && !ctx->recon) {
    if (loop) return t > 5 ? 1 : 8;
    return t > (pair ? 8.4 : 9) && t <= 10 ? 1 : 8;
  }
  if (prec == SQCG_F32) {
    if (t <= 2) return t <= 0.75 ? 8 : 4;
    if (!ctx->eightway || loop) return 1;
    return pair ? (t <= 4.45 ? 4 : 1) : t <= 2.5 || (t > 8 && t <= 9) ? 4 : 1;
  }
  if (t <= 0.5) return 8;
  if (prec == SQCG_FF) return t <= 5 || (t > 8 && t <= 10) ? 4 : 1;
  if (t > 5 || (t > 1.5 && ceil(t) - t <= 0.16)) return 1;
  return loop && t > 1.65 && t <= 1.8 ? 8 : 4;
}

int launch_dslash(sqcg_ctx* ctx, const DslashLaunch& L, cudaStream_t s) {
  if (!ctx->have_links) return SQCG_ERR_NO_LINKS;
  if (L.out_parity != 0 && L.out_parity != 1) return SQCG_ERR_INVALID_ARG;
  if (L.epi == EPI_TRUE_RESID) {
    if (L.prec != SQCG_F64 || !L.b || !L.y) return SQCG_ERR_INVALID_ARG;
    return L.out_prec == SQCG_F64 ? launch_r<double, double>(ctx, L, s) : launch_r<double, float>(ctx, L, s);
  }
  if (L.out_prec != L.prec) return SQCG_ERR_INVALID_ARG;
  if ((L.epi == EPI_NORMAL || L.epi == EPI_NORMAL_DOT || L.epi == EPI_SR_DOTS || L.epi == EPI_SR_DOTS2) && !L.y)
    return SQCG_ERR_INVALID_ARG;
  if (L.epi == EPI_SR_DOTS && !L.y3) return SQCG_ERR_INVALID_ARG;
  if (L.prec == SQCG_F64) return launch_r<double, double>(ctx, L, s);
  if (L.prec == SQCG_F32) return launch_r<float, float>(ctx, L, s);
  return SQCG_ERR_INVALID_ARG;
}
