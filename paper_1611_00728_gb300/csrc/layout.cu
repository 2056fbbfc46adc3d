// Host <-> device layout: links from the MILC forward-only AoS order into the
// parity-split structure of arrays [parity][mu][elem][Vh] (FP64 and FP32
// copies, phases folded), and colour vectors between host parity order
// [Vh][3] and device [3][Vh]. The paper's own layout is an x86 AoSoA with
// 8-way links (Sec. 3); on the GPU a site-index-fastest SoA gives coalesced
// warp loads instead.
#include <cmath>
#include <complex>

#include "ff_arith.cuh"
#include "sqcg_internal.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void coords_of(const Geom& g, long n, int& x, int& y, int& z, int& t) {
  x = (int)(n % g.Lx);
  n /= g.Lx;
  y = (int)(n % g.Ly);
  n /= g.Ly;
  z = (int)(n % g.Lz);
  t = (int)(n / g.Lz);
}

// raw[n][mu][9] (host link order) -> out64[par][mu][e][n/2] (e < 9), out32[par][mu][e][n/2] (e < nelem32: 9, or 6
// for the 12-real form) and the float-float copy outff, phases folded. A block takes 32 consecutive sites: their
// 18 KB are contiguous in raw, go through shared memory, and leave as runs of 16 sites per parity, direction
// and element. Bound by the FP64 pipe, which the conversions to FP32 run on (16^4: 29 us a field; the first form,
// with a thread reading its link's 144 bytes at a stride of 144 and a second pass for outff, took 61).
constexpr int kPackSites = 32, kPackThreads = 128;
__global__ void __launch_bounds__(kPackThreads) k_pack_links(const double2* __restrict__ raw, Geom g, int fold, int hop,
                                                             int nelem32, double2* __restrict__ out64,
                                                             float2* __restrict__ out32, float4* __restrict__ outff) {
  __shared__ double2 sm[kPackSites][37];  // 36 elements a site, padded against bank conflicts
  const long V = 2L * g.Vh, n0 = (long)blockIdx.x * kPackSites;
  const int ns = V - n0 < kPackSites ? (int)(V - n0) : kPackSites;
  for (int j = threadIdx.x; j < ns * 36; j += kPackThreads) sm[j / 36][j % 36] = raw[n0 * 36 + j];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int p = lane >> 4;  // parity; the half index of the site is ih
  const long ih = (n0 >> 1) + (lane & 15);
  if (2 * (lane & 15) >= ns) return;
  int x, y, z, t;
  coords_of(g, 2 * ih, x, y, z, t);
  const int odd = (y + z + t + p) & 1;  // 2 ih has x even
  x += odd;
  const int local = 2 * (lane & 15) + odd;
  for (int k = warp; k < 36; k += kPackThreads / 32) {
    const int mu = k / 9, e = k % 9;
    bool neg = false;
    if (fold) {
      const int c = (mu == 0) ? 0 : (mu == 1) ? x : (mu == 2) ? x + y : x + y + z;
      neg = c & 1;
      if (mu == 3 && g.apbc && t + hop >= g.Lt) neg = !neg;
    }
    double2 v = sm[local][k];
    if (neg) v = make_double2(-v.x, -v.y);
    const size_t at64 = (((size_t)p * 4 + mu) * 9 + e) * g.Vh + ih;
    const float4 f = split_ff(v);
    out64[at64] = v;
    outff[at64] = f;
    if (e < nelem32) out32[(((size_t)p * 4 + mu) * nelem32 + e) * g.Vh + ih] = make_float2(f.x, f.z);
  }
}

// Is every long link s W with W in SU(3) and s the one real scale s0, to 1e-12? With the phases folded by the
// caller, s carries eta_mu(n) and the boundary sign, which are divided out before it is compared. *bad is set
// where not. One thread a link, the block's links staged through shared memory.
constexpr int kCheckThreads = 128;
__global__ void __launch_bounds__(kCheckThreads) k_recon_check(const double2* __restrict__ raw, Geom g, int folded,
                                                               double s0, int* __restrict__ bad) {
  __shared__ double2 sm[kCheckThreads * 9];
  const long nlinks = 8L * g.Vh, l0 = (long)blockIdx.x * kCheckThreads;
  const int nl = nlinks - l0 < kCheckThreads ? (int)(nlinks - l0) : kCheckThreads;
  for (int j = threadIdx.x; j < nl * 9; j += kCheckThreads) sm[j] = raw[l0 * 9 + j];
  __syncthreads();
  if ((int)threadIdx.x >= nl) return;
  double2 U[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) U[e] = sm[threadIdx.x * 9 + e];
  auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
  double2 det = make_double2(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double2 m1 = mul(U[3 + (j + 1) % 3], U[6 + (j + 2) % 3]), m2 = mul(U[3 + (j + 2) % 3], U[6 + (j + 1) % 3]);
    const double2 d = mul(U[j], make_double2(m1.x - m2.x, m1.y - m2.y));
    det.x += d.x;
    det.y += d.y;
  }
  const double s = cbrt(det.x), s2 = s * s;
  const bool far = !(s2 > 1e-100 && s2 < 1e100);  // squares of the products below may leave the range of FP64
  bool ok = fabs(s) > 0.0 && isfinite(s) && fabs(det.y) <= 1e-12 * fabs(s2 * s);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) {
      double re = (a == b) ? -s2 : 0.0, im = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double2 u = U[a * 3 + c], v = U[b * 3 + c];
        re += u.x * v.x + u.y * v.y;
        im += u.y * v.x - u.x * v.y;
      }
      ok = ok && (far ? hypot(re, im) <= 1e-12 * s2 : re * re + im * im <= 1e-24 * s2 * s2);  // false for a NaN
    }
  double f = 1.0;
  if (folded) {
    const long l = l0 + threadIdx.x;
    const int mu = (int)(l & 3);
    int x, y, z, t;
    coords_of(g, l >> 2, x, y, z, t);
    const int e = (mu == 0) ? 0 : (mu == 1) ? x : (mu == 2) ? x + y : x + y + z;
    if (e & 1) f = -f;
    if (mu == 3 && g.apbc && t + 3 >= g.Lt) f = -f;
  }
  ok = ok && fabs(s * f - s0) <= 1e-12 * fabs(s0);
  if (!ok) *bad = 1;
}

// host parity order [Vh][3] complex double -> device [3][Vh] (FP64 or FP32)
template <typename O2>
__global__ void k_aos_to_soa(const double2* __restrict__ aos, O2* __restrict__ soa, int Vh) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Vh) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 v = aos[(size_t)i * 3 + c];
    O2 o;
    o.x = v.x;
    o.y = v.y;
    soa[(size_t)c * Vh + i] = o;
  }
}

// host parity order [Vh][3] complex double -> device [3][Vh] float-float (hi = fl32(v), lo = fl32(v - hi))
__global__ void k_aos_to_soa_ff(const double2* __restrict__ aos, float4* __restrict__ soa, int Vh) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Vh) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) soa[(size_t)c * Vh + i] = split_ff(aos[(size_t)i * 3 + c]);
}

__global__ void k_soa_ff_to_aos(const float4* __restrict__ soa, double2* __restrict__ aos, int Vh) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Vh) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 v = soa[(size_t)c * Vh + i];
    aos[(size_t)i * 3 + c] = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
  }
}

template <typename I2>
__global__ void k_soa_to_aos(const I2* __restrict__ soa, double2* __restrict__ aos, int Vh) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Vh) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const I2 v = soa[(size_t)c * Vh + i];
    aos[(size_t)i * 3 + c] = make_double2((double)v.x, (double)v.y);
  }
}

template <typename I2, typename O2>
__global__ void k_convert(const I2* __restrict__ in, O2* __restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const I2 v = in[i];
  O2 o;
  o.x = v.x;
  o.y = v.y;
  out[i] = o;
}

// 8-way FP32 backward links: out[p][mu][e][n_h] = -(U_mu(n - d mu))^dagger, from the
// folded FP64 forward links; e < nelem (6: first two rows for the 12-real form)
__global__ void k_pack_backward(const double2* __restrict__ fwd64, Geom g, int d, int nelem, float2* __restrict__ out) {
  const long V = 2L * g.Vh;
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= 4 * V) return;
  const int mu = (int)(tid / V);
  const long n = tid % V;
  int c[4];
  long m = n;
  c[0] = (int)(m % g.Lx); m /= g.Lx;
  c[1] = (int)(m % g.Ly); m /= g.Ly;
  c[2] = (int)(m % g.Lz);
  c[3] = (int)(m / g.Lz);
  const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
  const int Ls[4] = {g.Lx, g.Ly, g.Lz, g.Lt};
  int cb[4] = {c[0], c[1], c[2], c[3]};
  cb[mu] = ((c[mu] - d) % Ls[mu] + Ls[mu]) % Ls[mu];
  const long nb = cb[0] + (long)g.Lx * (cb[1] + (long)g.Ly * (cb[2] + (long)g.Lz * cb[3]));
  const int q = 1 - par;
  const size_t src = ((size_t)q * 4 + mu) * 9 * g.Vh + (nb >> 1);
  const size_t dst = ((size_t)par * 4 + mu) * nelem * g.Vh + (n >> 1);
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) {
      const int e = a * 3 + b;
      if (e >= nelem) continue;
      const double2 u = fwd64[src + (size_t)(b * 3 + a) * g.Vh];  // element (b, a) of the forward link
      out[dst + (size_t)e * g.Vh] = make_float2(__double2float_rn(-u.x), __double2float_rn(u.y));
    }
}

// The scale of the first long link (site 0, direction x: its phase and boundary sign are 1): cbrt(Re det).
double first_link_scale(const double* p) {
  typedef std::complex<double> cd;
  cd U[3][3];
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) U[a][b] = cd(p[(a * 3 + b) * 2], p[(a * 3 + b) * 2 + 1]);
  const cd det = U[0][0] * (U[1][1] * U[2][2] - U[1][2] * U[2][1]) -
                 U[0][1] * (U[1][0] * U[2][2] - U[1][2] * U[2][0]) +
                 U[0][2] * (U[1][0] * U[2][1] - U[1][1] * U[2][0]);
  return std::cbrt(det.real());
}

// 12-real eligibility of long links in device memory (host link order); first: its first link in host memory
int recon_check(sqcg_ctx* ctx, const double2* lng, const double* first, double* s0_out) {
  const double s0 = first_link_scale(first);
  if (!(std::fabs(s0) > 0.0) || !std::isfinite(s0)) return SQCG_ERR_RECON_REJECTED;
  int* bad = nullptr;
  if (cudaMalloc((void**)&bad, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return SQCG_ERR_NO_MEMORY;
  }
  cudaStream_t s = ctx->stream;
  int h = 0;
  const long nlinks = 8L * ctx->g.Vh;
  cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    k_recon_check<<<(unsigned)((nlinks + kCheckThreads - 1) / kCheckThreads), kCheckThreads, 0, s>>>(
        lng, ctx->g, (ctx->flags & SQCG_PHASES_FOLDED) ? 1 : 0, s0, bad);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(bad);
  if (e != cudaSuccess) {
    sqcg_set_last_cuda_error(e, "long-link check", __FILE__, __LINE__);
    return SQCG_ERR_CUDA;
  }
  *s0_out = s0;
  return h ? SQCG_ERR_RECON_REJECTED : SQCG_OK;
}

void free_stage(sqcg_ctx* ctx) {
  cudaFree(ctx->stage);
  ctx->stage = nullptr;
  ctx->stage_bytes = 0;
}

int ensure_stage(sqcg_ctx* ctx, size_t bytes) {
  if (ctx->stage_bytes >= bytes) return SQCG_OK;
  free_stage(ctx);
  if (cudaMalloc(&ctx->stage, bytes) != cudaSuccess) {
    cudaGetLastError();
    return SQCG_ERR_NO_MEMORY;
  }
  ctx->stage_bytes = bytes;
  return SQCG_OK;
}

}  // namespace

namespace {

// staging of host links up to this size stays with the context, larger staging lives for the call
constexpr size_t kKeptStage = (size_t)64 << 20;

void free_links(sqcg_ctx* ctx) {
  cudaFree(ctx->fat64); cudaFree(ctx->lng64); cudaFree(ctx->fat32); cudaFree(ctx->lng32);
  cudaFree(ctx->fatb32); cudaFree(ctx->lngb32);
  cudaFree(ctx->fatff); cudaFree(ctx->lngff);
  ctx->fat64 = ctx->lng64 = nullptr;
  ctx->fat32 = ctx->lng32 = nullptr;
  ctx->fatb32 = ctx->lngb32 = nullptr;
  ctx->fatff = ctx->lngff = nullptr;
}

// Device link arrays for 12-real or full long links, with the backward arrays of the 8-way form or without; those
// of the links before are kept where they are the same (an allocation of this size takes 0.1 ms and more).
int ensure_links(sqcg_ctx* ctx, int nl32, bool eightway) {
  const size_t Vh = ctx->g.Vh, n9 = 2 * 4 * 9 * Vh, nl = 2 * 4 * (size_t)nl32 * Vh;
  if (ctx->fat64 && ctx->link_nl32 != nl32) free_links(ctx);
  if (!eightway) {
    cudaFree(ctx->fatb32); cudaFree(ctx->lngb32);
    ctx->fatb32 = ctx->lngb32 = nullptr;
  }
  auto want = [](auto** p, size_t bytes) { return *p || cudaMalloc((void**)p, bytes) == cudaSuccess; };
  const bool ok = want(&ctx->fat64, n9 * sizeof(double2)) && want(&ctx->lng64, n9 * sizeof(double2)) &&
                  want(&ctx->fat32, n9 * sizeof(float2)) && want(&ctx->lng32, nl * sizeof(float2)) &&
                  want(&ctx->fatff, n9 * sizeof(float4)) && want(&ctx->lngff, n9 * sizeof(float4)) &&
                  (!eightway || (want(&ctx->fatb32, n9 * sizeof(float2)) && want(&ctx->lngb32, nl * sizeof(float2))));
  if (!ok) {
    cudaGetLastError();
    free_links(ctx);
    return SQCG_ERR_NO_MEMORY;
  }
  ctx->link_nl32 = nl32;
  return SQCG_OK;
}

// fat, lng: host order [V][4][3][3] complex, in host memory or (on_device) in device memory.
// What earlier calls queued on this stream is over before a kept array or the staging is written again. Work that
// they left on another stream may still be reading: where the context has been on several, both are given back and
// allocated anew instead (the runtime frees memory only once nothing on the device uses it; that also holds for
// streams that are gone or being captured, which nothing here could wait for).
int load_links(sqcg_ctx* ctx, const double* fat, const double* lng, int opts, bool on_device) {
  if (!fat || !lng) return SQCG_ERR_INVALID_ARG;
  if (opts & ~(SQCG_RECON12_LONG | SQCG_EIGHT_WAY)) return SQCG_ERR_INVALID_ARG;
  const bool recon = (opts & SQCG_RECON12_LONG) != 0;
  const bool eightway = (opts & SQCG_EIGHT_WAY) != 0;
  cudaStream_t s = ctx->stream;
  const size_t V = 2 * (size_t)ctx->g.Vh, bytes = V * 4 * 9 * sizeof(double2);

  // host links are staged one field at a time, the long ones first: a rejection of the 12-real form leaves
  // the earlier links as they are
  void* own = nullptr;
  void* raw = nullptr;
  if (!on_device) {
    if (bytes <= kKeptStage) {
      if (ctx->streams_mixed) free_stage(ctx);
      SQCG_TRY(ensure_stage(ctx, bytes));
      raw = ctx->stage;
    } else if (cudaMalloc(&own, bytes) != cudaSuccess) {
      cudaGetLastError();
      return SQCG_ERR_NO_MEMORY;
    } else {
      raw = own;
    }
  }
  double s0 = 1.0;
  int rc = SQCG_OK;
  const double2* src = (const double2*)lng;
  if (!on_device) {
    if (cudaMemcpyAsync(raw, lng, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) rc = SQCG_ERR_CUDA;
    src = (const double2*)raw;
  }
  if (rc == SQCG_OK && recon) {
    double first[18];
    const double* f = lng;
    if (on_device) {
      if (cudaMemcpyAsync(first, lng, sizeof(first), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        rc = SQCG_ERR_CUDA;
      f = first;
    }
    if (rc == SQCG_OK) rc = recon_check(ctx, src, f, &s0);
  }
  if (rc != SQCG_OK) {
    if (rc == SQCG_ERR_CUDA) sqcg_set_last_cuda_error(cudaGetLastError(), "load_links", __FILE__, __LINE__);
    cudaFree(own);
    return rc;
  }

  // the 12-real form is used for the FP32 copy only: on this GPU the FP64 Dslash is
  // bound by FP64 arithmetic, which rebuilding the third row would only add to
  const int nl32 = recon ? 6 : 9;
  // drop earlier links
  if (cudaStreamSynchronize(s) != cudaSuccess) rc = SQCG_ERR_CUDA;
  ctx->eightway = false;
  ctx->have_links = false;
  free_graphs(ctx);
  free_batch_plan(ctx);
  if (ctx->streams_mixed) {
    free_links(ctx);
    if (on_device) free_stage(ctx);  // host links: done above, or staged elsewhere
    ctx->streams_mixed = false;
  }
  if (rc == SQCG_OK) rc = ensure_links(ctx, nl32, eightway);
  const int fold = (ctx->flags & SQCG_PHASES_FOLDED) ? 0 : 1;
  const unsigned grid = (unsigned)((V + kPackSites - 1) / kPackSites);
  if (rc == SQCG_OK) {
    k_pack_links<<<grid, kPackThreads, 0, s>>>(src, ctx->g, fold, 3, nl32, ctx->lng64, ctx->lng32, ctx->lngff);
    src = (const double2*)fat;
    // the long pass must finish reading the staging buffer before it is overwritten (same stream)
    if (cudaGetLastError() != cudaSuccess ||
        (!on_device && cudaMemcpyAsync(raw, fat, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess))
      rc = SQCG_ERR_CUDA;
    if (!on_device) src = (const double2*)raw;
  }
  if (rc == SQCG_OK) {
    k_pack_links<<<grid, kPackThreads, 0, s>>>(src, ctx->g, fold, 1, 9, ctx->fat64, ctx->fat32, ctx->fatff);
    if (eightway) {
      const unsigned gb = (unsigned)((4 * V + kThreads - 1) / kThreads);
      k_pack_backward<<<gb, kThreads, 0, s>>>(ctx->fat64, ctx->g, 1, 9, ctx->fatb32);
      k_pack_backward<<<gb, kThreads, 0, s>>>(ctx->lng64, ctx->g, 3, nl32, ctx->lngb32);
    }
    if (cudaGetLastError() != cudaSuccess) rc = SQCG_ERR_CUDA;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) rc = SQCG_ERR_CUDA;
  if (rc == SQCG_ERR_CUDA) sqcg_set_last_cuda_error(cudaGetLastError(), "load_links", __FILE__, __LINE__);
  cudaFree(own);
  if (rc != SQCG_OK) return rc;
  ctx->eightway = eightway;
  ctx->recon = recon;
  ctx->long_scale = s0;
  ctx->have_links = true;
  static unsigned long long generation = 0;
  ctx->links_gen = __atomic_add_fetch(&generation, 1ULL, __ATOMIC_RELAXED);
  return SQCG_OK;
}

}  // namespace

int layout_load_links(sqcg_ctx* ctx, const double* fat, const double* lng, int opts) {
  return load_links(ctx, fat, lng, opts, false);
}

int layout_load_links_device(sqcg_ctx* ctx, const double* fat, const double* lng, int opts) {
  return load_links(ctx, fat, lng, opts, true);
}

int layout_pack_spinor(sqcg_ctx* ctx, int prec, const double* host, void* dev) {
  if (!host || !dev || (prec != SQCG_F64 && prec != SQCG_F32 && prec != SQCG_FF)) return SQCG_ERR_INVALID_ARG;
  const int Vh = ctx->g.Vh;
  const size_t bytes = (size_t)Vh * 3 * sizeof(double2);
  SQCG_TRY(ensure_stage(ctx, bytes));
  cudaStream_t s = ctx->stream;
  SQCG_CUDA_TRY(cudaMemcpyAsync(ctx->stage, host, bytes, cudaMemcpyHostToDevice, s));
  if (prec == SQCG_F64)
    k_aos_to_soa<double2><<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const double2*)ctx->stage, (double2*)dev, Vh);
  else if (prec == SQCG_FF)
    k_aos_to_soa_ff<<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const double2*)ctx->stage, (float4*)dev, Vh);
  else
    k_aos_to_soa<float2><<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const double2*)ctx->stage, (float2*)dev, Vh);
  SQCG_CUDA_TRY(cudaGetLastError());
  return SQCG_OK;
}

int layout_unpack_spinor(sqcg_ctx* ctx, int prec, const void* dev, double* host) {
  if (!host || !dev || (prec != SQCG_F64 && prec != SQCG_F32 && prec != SQCG_FF)) return SQCG_ERR_INVALID_ARG;
  const int Vh = ctx->g.Vh;
  const size_t bytes = (size_t)Vh * 3 * sizeof(double2);
  SQCG_TRY(ensure_stage(ctx, bytes));
  cudaStream_t s = ctx->stream;
  if (prec == SQCG_F64)
    k_soa_to_aos<double2><<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const double2*)dev, (double2*)ctx->stage, Vh);
  else if (prec == SQCG_FF)
    k_soa_ff_to_aos<<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const float4*)dev, (double2*)ctx->stage, Vh);
  else
    k_soa_to_aos<float2><<<grid_for(Vh, kThreads), kThreads, 0, s>>>((const float2*)dev, (double2*)ctx->stage, Vh);
  SQCG_CUDA_TRY(cudaGetLastError());
  SQCG_CUDA_TRY(cudaMemcpyAsync(host, ctx->stage, bytes, cudaMemcpyDeviceToHost, s));
  SQCG_CUDA_TRY(cudaStreamSynchronize(s));
  return SQCG_OK;
}

int layout_convert(sqcg_ctx* ctx, int from_prec, const void* src, int to_prec, void* dst, cudaStream_t s) {
  const int n = ctx->g.Vh * 3;
  const int grid = grid_for(n, kThreads);
  if (from_prec == SQCG_F64 && to_prec == SQCG_F32)
    k_convert<double2, float2><<<grid, kThreads, 0, s>>>((const double2*)src, (float2*)dst, n);
  else if (from_prec == SQCG_F32 && to_prec == SQCG_F64)
    k_convert<float2, double2><<<grid, kThreads, 0, s>>>((const float2*)src, (double2*)dst, n);
  else if (from_prec == to_prec)
    SQCG_CUDA_TRY(cudaMemcpyAsync(dst, src, (size_t)n * (from_prec == SQCG_F64 ? 16 : 8), cudaMemcpyDeviceToDevice, s));
  else
    return SQCG_ERR_INVALID_ARG;
  SQCG_CUDA_TRY(cudaGetLastError());
  return SQCG_OK;
}

unsigned long long sqcg_links_generation(const sqcg_ctx* ctx) { return ctx->links_gen; }
