// HISQ link construction on the GPU: thin links -> fat and long links in FP64.
//
// The paper's benchmark application evolves the HISQ action (Sec. 4), whose CG
// consumes these links; the construction is that of the HISQ action (Follana
// et al., hep-lat/0610092):
//   V = smear(U, level 1)  one link + 3-, 5-, 7-link staples (fat7)
//   W = V (V^+ V)^(-1/2)   U(3) projection
//   fat = smear(W, level 2) the same staples + the Lepage 5-link staple
//   long = naik W_mu(n) W_mu(n+mu) W_mu(n+2mu)
// Links are unphased and periodic; the staggered phases and the time-boundary
// sign are folded in afterwards, when the result is loaded into a context.
//
// One smearing level is three kernels over full-lattice structure-of-arrays
// fields [field][element][V] (site fastest, coalesced):
//   A: S^s_{mu nu}(n), the single-sign 3-staples (24 fields; only where the level
//      has a Lepage term), and their sums S3_{mu nu} = S^+ + S^- (12 fields);
//   B: Z_{mu nu}(n) = c5 (S3_{mu rho} + S3_{mu sig})(n)
//                    + c7 (wrap_rho S3_{mu sig} + wrap_sig S3_{mu rho})(n),
//      {rho, sig} the two directions other than mu, nu; with a Lepage term
//      Y^s = Z + cL S^s, which takes the place of S^s;
//   C: F_mu(n) = c1 U_mu(n) + sum_nu [ c3 S3_{mu nu}(n) + sum_s wrap^s_nu(Y^s_{mu nu})(n) ]
//      (Y^s = Z without a Lepage term),
// where wrap^+_d X (n) = U_d(n) X(n+d) U_d(n+mu)^+ and
//       wrap^-_d X (n) = U_d(n-d)^+ X(n-d) U_d(n-d+mu).
// Expanding C gives every 5-link staple (outer nu, inner rho) with c5, every
// 7-link staple (outer nu, middle rho, inner sig) with c7 and every Lepage
// staple (nu twice, same sign) with cL, at 48 3x3 products per link per level
// (12 in A, 24 in B, 12 in C).
//
// Arithmetic: on this GPU an FP64 FMA issues at 1/64 of the FP32 rate, and the FP64 version of these
// kernels ran with the FP64 pipe 90-97% busy. The staple products therefore run in float-float
// arithmetic: every real is an unevaluated sum hi + lo of two floats (48-bit significand), and products
// accumulate by error-free transformations on the FP32 pipe. The fields in the workspace hold a complex
// number as the pairs (re_hi, im_hi) and (re_lo, im_lo), 16 bytes like a double2: re and im go through the
// same operations, so every step is one packed two-lane FP32 instruction (sm_100 and later):
//   TwoProduct(a, b) = (p, e): p = fl(a b), e = fma(a, b, -p)   exact (Dekker 1971, with an FMA)
//   TwoSum(s, p) = (s', t): s' = fl(s + p), v = s' - s, t = (s - (s' - v)) + (p - v)   exact (Knuth, TAOCP
//                  vol. 2, 4.2.2)
// with e, t and the cross terms a_lo b and a b_lo in the low word. (Summing with s' = fma(a, b, s) instead saves three
// instructions in twelve but is not exact where s and a b cancel: their difference can need more than 24 bits.)
// The thin links are split at the first kernel, the U(3) projection divides in FP64, and the outputs are
// joined back to FP64.
//
// A thread computes one row of a matrix: row i of a product needs row i of the left factor only, and both
// products of a wrap keep their rows. With whole matrices in a thread these kernels took 168-232 registers, so that
// 12-24% of the warp slots hid the latency of the accumulation chains (FMA pipe 52-60% busy). A block is 64 sites
// x 3 rows, so the right factors that three threads read come from L1 for two of them. 24^3 x 32: 12.8 -> 9.9 ms,
// the packed instructions (two pipe slots each) filling 71% of the FMA pipe (profiles/hisq_smear_32x32x32x32.md); kernel A 1.33 -> 1.06 ms, B 2.63 -> 2.12,
// C 1.66 -> 1.14 (level 1), at 5, 4 and 4 blocks a SM (one fewer each: 10.9 ms; five for all: 10.0).
#include <math.h>
#include <string.h>

#include "ff_arith.cuh"
#include "sqcg_internal.cuh"

namespace {

constexpr int kThreads = 128;

struct Lat {
  int L[4];
  long V;
};

// ---- packed float-float complex numbers ----
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pk(float x, float y) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 upk(f32x2 a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

struct __align__(16) C2 {  // complex: (re, im) high and low words
  f32x2 h, l;
};
__device__ __forceinline__ C2 czero() { return {0ull, 0ull}; }
__device__ __forceinline__ C2 cswap(C2 a) {  // (im, re)
  const float2 h = upk(a.h), l = upk(a.l);
  return {pk(h.y, h.x), pk(l.y, l.x)};
}
__device__ __forceinline__ C2 from_double(double2 v) {
  const float4 f = split_ff(v);
  return {pk(f.x, f.z), pk(f.y, f.w)};
}
__device__ __forceinline__ double2 to_double(C2 a) {
  const float2 h = upk(a.h), l = upk(a.l);
  return make_double2((double)h.x + (double)l.x, (double)h.y + (double)l.y);
}

// fl(a b). Written as an FMA with zero: with mul.rn.f32x2, the addition that takes its result came out as one FMA for
// all of 65536 random operands (CUDA 13.0; in 14121 of them that is another number than the two roundings give), with
// this form as two roundings for all. Rounded once, the error terms below would be those of another sum, and the links
// off by some 1e-8, which the tests' 1e-12 shows.
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { return fma2(a, b, 0ull); }

// acc += a b lane by lane, a = (ah, al), na = -ah, b = (bh, bl); the low word is not renormalised in between
__device__ __forceinline__ void acc2(C2& acc, f32x2 ah, f32x2 na, f32x2 al, C2 b) {
  const f32x2 np = mul2(na, b.h);  // -p
  const f32x2 e = fma2(ah, b.l, fma2(al, b.h, fma2(ah, b.h, np)));
  const f32x2 s = sub2(acc.h, np);
  const f32x2 v = sub2(s, acc.h);
  const f32x2 t = sub2(sub2(acc.h, sub2(s, v)), add2(np, v));
  acc.l = add2(acc.l, add2(t, e));
  acc.h = s;
}
// acc = a b
__device__ __forceinline__ void first2(C2& acc, f32x2 ah, f32x2 na, f32x2 al, C2 b) {
  acc.h = mul2(ah, b.h);
  acc.l = fma2(ah, b.l, fma2(al, b.h, fma2(ah, b.h, mul2(na, b.h))));
}
__device__ __forceinline__ void cnorm(C2& a) {
  const f32x2 s = add2(a.h, a.l);
  a.l = sub2(a.l, sub2(s, a.h));
  a.h = s;
}
// a += b, renormalised
__device__ __forceinline__ void cadd(C2& a, C2 b) {
  const f32x2 s = add2(a.h, b.h);
  const f32x2 v = sub2(s, a.h);
  f32x2 e = add2(sub2(a.h, sub2(s, v)), sub2(b.h, v));
  e = add2(e, add2(a.l, b.l));
  a.h = add2(s, e);
  a.l = sub2(e, sub2(a.h, s));
}

// The left operand of products, its components spread over the lanes with the signs of the form:
// PLAIN a b, CONJ_L a^* b, CONJ_R a b^*
enum Form { PLAIN = 0, CONJ_L = 1, CONJ_R = 2 };
struct Left {
  f32x2 rh, nrh, rl, ih, nih, il;  // nrh = -rh, nih = -ih
};
template <Form F>
__device__ __forceinline__ Left left(C2 a) {
  const float2 h = upk(a.h), l = upk(a.l);
  if (F == PLAIN)
    return {pk(h.x, h.x), pk(-h.x, -h.x), pk(l.x, l.x), pk(-h.y, h.y), pk(h.y, -h.y), pk(-l.y, l.y)};
  if (F == CONJ_L)
    return {pk(h.x, h.x), pk(-h.x, -h.x), pk(l.x, l.x), pk(h.y, -h.y), pk(-h.y, h.y), pk(l.y, -l.y)};
  return {pk(h.x, -h.x), pk(-h.x, h.x), pk(l.x, -l.x), pk(h.y, h.y), pk(-h.y, -h.y), pk(l.y, l.y)};
}
template <bool FIRST = false>
__device__ __forceinline__ void cmac(C2& acc, const Left& a, C2 b) {
  if (FIRST) first2(acc, a.rh, a.nrh, a.rl, b);
  else acc2(acc, a.rh, a.nrh, a.rl, b);
  acc2(acc, a.ih, a.nih, a.il, cswap(b));
}
// acc += c a for a float-float real c
__device__ __forceinline__ void caxpy(C2& acc, float2 c, C2 a) {
  acc2(acc, pk(c.x, c.x), pk(-c.x, -c.x), pk(c.y, c.y), a);
  cnorm(acc);
}

struct R3 {  // a row
  C2 e[3];
};
__device__ __forceinline__ R3 rzero() {
  R3 r;
#pragma unroll
  for (int j = 0; j < 3; ++j) r.e[j] = czero();
  return r;
}

// element k of field f at site n: fields [f][e][V]
__device__ __forceinline__ C2 ld(const C2* __restrict__ f, long V, long n, int e) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(f + (size_t)e * V + n));
  return {v.x, v.y};
}
__device__ __forceinline__ const C2* field(const C2* base, int k, long V) { return base + (size_t)k * 9 * V; }
__device__ __forceinline__ R3 ld_row(const C2* __restrict__ f, long V, long n, int i) {
  R3 r;
#pragma unroll
  for (int j = 0; j < 3; ++j) r.e[j] = ld(f, V, n, 3 * i + j);
  return r;
}
__device__ __forceinline__ void st_row(C2* f, long V, long n, int i, const R3& r) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
    *reinterpret_cast<ulonglong2*>(f + (size_t)(3 * i + j) * V + n) = make_ulonglong2(r.e[j].h, r.e[j].l);
}

// acc += row i of A X (FIRST: acc = ...): a[k] = A_ik
template <Form F, bool FIRST = false>
__device__ __forceinline__ void row_mul(R3& acc, const R3& a, const C2* __restrict__ X, long V, long n) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Left l = left<F>(a.e[k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (FIRST && k == 0) cmac<true>(acc.e[j], l, ld(X, V, n, 3 * k + j));
      else cmac(acc.e[j], l, ld(X, V, n, 3 * k + j));
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) cnorm(acc.e[j]);
}
// acc += (row a) B^+
__device__ __forceinline__ void row_mul_dag(R3& acc, const R3& a, const C2* __restrict__ B, long V, long n) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Left l = left<CONJ_R>(a.e[k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) cmac(acc.e[j], l, ld(B, V, n, 3 * j + k));
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) cnorm(acc.e[j]);
}

// A direction at a site: index offset of the neighbour k steps on (periodic, |k| < L)
struct Dir {
  int c, L;
  long st;
  __device__ __forceinline__ long off(int k) const {
    const int x = c + k;
    return (x >= L ? k - L : x < 0 ? k + L : k) * st;
  }
};
__device__ __forceinline__ Dir dir_of(const Lat& g, long n, int d) {
  const long st = d == 0 ? 1 : d == 1 ? g.L[0] : d == 2 ? (long)g.L[0] * g.L[1] : (long)g.L[0] * g.L[1] * g.L[2];
  const int L = d == 0 ? g.L[0] : d == 1 ? g.L[1] : d == 2 ? g.L[2] : g.L[3];
  return {(int)((n / st) % L), L, st};
}
// the i-th direction other than mu (increasing order), and the inverse
__device__ __forceinline__ int other(int mu, int i) { return i + (i >= mu ? 1 : 0); }
__device__ __forceinline__ int other_index(int mu, int d) { return d - (d > mu ? 1 : 0); }
// staple fields: single-sign S^s_{mu d} at (mu*3 + index of d)*2 + s, their sum S3_{mu d} at 24 + mu*3 + index
constexpr int kNumS = 36;
__device__ __forceinline__ int s3_field(int mu, int d) { return 24 + mu * 3 + other_index(mu, d); }

// acc += row i of wrap^s_d X at n, X a field in direction mu
__device__ __forceinline__ void wrap_row(R3& acc, const C2* __restrict__ U, long V, long n, const Dir& dmu, const Dir& dd,
                                         int d, int s, const C2* __restrict__ X, int i) {
  const C2* Ud = field(U, d, V);
  if (s == 0) {
    R3 m;
    row_mul<PLAIN, true>(m, ld_row(Ud, V, n, i), X, V, n + dd.off(1));
    row_mul_dag(acc, m, Ud, V, n + dmu.off(1));
  } else {
    const long y = n + dd.off(-1);
    R3 a, m;
#pragma unroll
    for (int k = 0; k < 3; ++k) a.e[k] = ld(Ud, V, y, 3 * k + i);
    row_mul<CONJ_L, true>(m, a, X, V, y);
    row_mul<PLAIN>(acc, m, Ud, V, y + dmu.off(1));
  }
}

// threads of the staple kernels: sites x rows
constexpr int kSites = 64;

// host AoS [V][4][9] (FP64) -> [mu][e][V] (float-float)
__global__ void __launch_bounds__(kThreads) k_links_to_fields(Lat g, const double2* __restrict__ aos,
                                                              C2* __restrict__ U) {
  const long n = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  const int mu = blockIdx.y;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const C2 v = from_double(aos[((size_t)n * 4 + mu) * 9 + e]);
    *reinterpret_cast<ulonglong2*>(U + ((size_t)mu * 9 + e) * g.V + n) = make_ulonglong2(v.h, v.l);
  }
}

// A: 3-staples S^+_{mu nu}, S^-_{mu nu} (s = 0 forward, 1 backward; written if `signs`) and S3_{mu nu} = S^+ + S^-
__global__ void __launch_bounds__(3 * kSites, 5) k_staple3(Lat g, const C2* __restrict__ U, C2* __restrict__ S, int signs) {
  const long n = (long)blockIdx.x * kSites + threadIdx.x, V = g.V;
  if (n >= V) return;
  const int i = threadIdx.y;
  const int f = blockIdx.y;  // mu*3 + nu index
  const int mu = f / 3, nu = other(mu, f % 3);
  const Dir dmu = dir_of(g, n, mu), dnu = dir_of(g, n, nu);
  const C2* X = field(U, mu, V);
  R3 sp = rzero(), sm = rzero();
  wrap_row(sp, U, V, n, dmu, dnu, nu, 0, X, i);
  wrap_row(sm, U, V, n, dmu, dnu, nu, 1, X, i);
  if (signs) {
    st_row(S + (size_t)(2 * f) * 9 * V, V, n, i, sp);
    st_row(S + (size_t)(2 * f + 1) * 9 * V, V, n, i, sm);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) cadd(sm.e[j], sp.e[j]);
  st_row(S + (size_t)(24 + f) * 9 * V, V, n, i, sm);
}

// B: Z_{mu nu} = c5 (S3_{mu rho} + S3_{mu sig}) + c7 (wrap_rho S3_{mu sig} + wrap_sig S3_{mu rho})
// (c5, c7 as float-float pairs; a zero coefficient skips its term); cL = 0: written to Z, else
// Y^s = Z + cL S^s in place of S^s
__global__ void __launch_bounds__(3 * kSites, 4) k_staple57(Lat g, const C2* __restrict__ U, C2* S, float2 c5, float2 c7,
                                                         float2 cL, C2* __restrict__ Z) {
  const long n = (long)blockIdx.x * kSites + threadIdx.x, V = g.V;
  if (n >= V) return;
  const int i = threadIdx.y;
  const int f = blockIdx.y;  // mu*3 + nu index
  const int mu = f / 3, nu = other(mu, f % 3);
  int rho = 0;
  while (rho == mu || rho == nu) ++rho;
  const int sig = 6 - mu - nu - rho;
  const C2* S3r = field(S, s3_field(mu, rho), V);
  const C2* S3s = field(S, s3_field(mu, sig), V);
  R3 z = rzero();
  if (c5.x != 0.f) {
    R3 t = ld_row(S3r, V, n, i);
    const R3 u = ld_row(S3s, V, n, i);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cadd(t.e[j], u.e[j]);
      caxpy(z.e[j], c5, t.e[j]);
    }
  }
  if (c7.x != 0.f) {
    const Dir dmu = dir_of(g, n, mu);
    R3 w = rzero();
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
      const int d = q == 0 ? rho : sig;
      const Dir dd = dir_of(g, n, d);
      const C2* X = q == 0 ? S3s : S3r;
      wrap_row(w, U, V, n, dmu, dd, d, 0, X, i);
      wrap_row(w, U, V, n, dmu, dd, d, 1, X, i);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) caxpy(z.e[j], c7, w.e[j]);
  }
  if (cL.x == 0.f) {
    st_row(Z + (size_t)f * 9 * V, V, n, i, z);
    return;
  }
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    C2* Y = S + (size_t)(2 * f + s) * 9 * V;
    R3 y = z;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Y + (size_t)(3 * i + j) * V + n);
      caxpy(y.e[j], cL, C2{v.x, v.y});
    }
    st_row(Y, V, n, i, y);
  }
}

// C: F_mu = c1 U_mu + sum_nu [ c3 S3_{mu nu} + sum_s wrap^s_nu Y^s_{mu nu} ], Y^s at Y + (f per_sign + s (per_sign - 1))
// fields for f = mu*3 + nu index: Z with per_sign = 1, the fields in place of S^s with 2; none if Y is null.
// out: float-float structure of arrays [mu][e][V], or FP64 in the host order [V][4][9] when aos != 0
__global__ void __launch_bounds__(3 * kSites, 4) k_smear_links(Lat g, const C2* __restrict__ U, const C2* __restrict__ S,
                                                            const C2* __restrict__ Y, int per_sign, float2 c1, float2 c3,
                                                            int aos, void* __restrict__ out) {
  const long n = (long)blockIdx.x * kSites + threadIdx.x, V = g.V;
  if (n >= V) return;
  const int i = threadIdx.y, mu = blockIdx.y;
  const Dir dmu = dir_of(g, n, mu);
  R3 F = rzero();
  {
    const R3 u = ld_row(field(U, mu, V), V, n, i);
#pragma unroll
    for (int j = 0; j < 3; ++j) caxpy(F.e[j], c1, u.e[j]);
  }
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    const int nu = other(mu, q), f = mu * 3 + q;
    if (c3.x != 0.f) {  // both signs: S3_{mu nu}
      const R3 t = ld_row(field(S, 24 + f, V), V, n, i);
#pragma unroll
      for (int j = 0; j < 3; ++j) caxpy(F.e[j], c3, t.e[j]);
    }
    if (Y) {
      const Dir dnu = dir_of(g, n, nu);
      const C2* Yf = field(Y, f * per_sign, V);
      wrap_row(F, U, V, n, dmu, dnu, nu, 0, Yf, i);
      wrap_row(F, U, V, n, dmu, dnu, nu, 1, field(Yf, per_sign - 1, V), i);
    }
  }
  if (aos) {
    double2* p = static_cast<double2*>(out) + ((size_t)n * 4 + mu) * 9 + 3 * i;
#pragma unroll
    for (int j = 0; j < 3; ++j) p[j] = to_double(F.e[j]);
  } else {
    st_row(static_cast<C2*>(out) + (size_t)mu * 9 * V, V, n, i, F);
  }
}

// ---- float-float 3x3 complex matrices with a thread each (the projection) ----
struct F3 {
  float4 e[9];
};
// acc += a b, acc += conj(a) b (float-float complex; the low words are not renormalised in between: fnorm
// after a few terms)
__device__ __forceinline__ void fcfma(float4& acc, float4 a, float4 b) {
  ff_acc(acc.x, acc.y, a.x, a.y, b.x, b.y);
  ff_acc(acc.x, acc.y, -a.z, -a.w, b.z, b.w);
  ff_acc(acc.z, acc.w, a.x, a.y, b.z, b.w);
  ff_acc(acc.z, acc.w, a.z, a.w, b.x, b.y);
}
__device__ __forceinline__ void fcfma_ca(float4& acc, float4 a, float4 b) {
  ff_acc(acc.x, acc.y, a.x, a.y, b.x, b.y);
  ff_acc(acc.x, acc.y, a.z, a.w, b.z, b.w);
  ff_acc(acc.z, acc.w, a.x, a.y, b.z, b.w);
  ff_acc(acc.z, acc.w, -a.z, -a.w, b.x, b.y);
}
__device__ __forceinline__ void fnorm(float4& v) {
  ff_norm(v.x, v.y);
  ff_norm(v.z, v.w);
}

// U(3) projection W = V (V^+ V)^(-1/2): the unitary polar factor of V, by Newton's
// iteration X <- (g X + X^{-+} / g) / 2 with Frobenius-norm scaling g while far from
// convergence (Higham, SIAM J. Sci. Stat. Comput. 7 (1986) 1160). X^{-+} is the
// conjugated cofactor matrix over conj(det X). At most kMaxPolar steps; a singular or
// non-finite link, or no convergence, sets *err and leaves the link as it is.
// The matrix arithmetic (cofactors, determinant, update) is float-float. Any g > 0 keeps the
// polar factor, so g comes from FP32 norms; X^{-+} must be exact to the working precision, so
// 1 / |det|^2 is one FP64 division on the joined value, split back. The step size is measured in
// FP32 from the float-float differences.
constexpr int kMaxPolar = 40;

__device__ __forceinline__ float4 fneg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }

__global__ void __launch_bounds__(kThreads) k_u3_project(Lat g, C2* __restrict__ F, int* __restrict__ err) {
  const long n = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  const int mu = blockIdx.y;
  F3 X;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const C2 v = ld(field(F, mu, g.V), g.V, n, e);
    const float2 h = upk(v.h), l = upk(v.l);
    X.e[e] = make_float4(h.x, l.x, h.y, l.y);
  }
  bool ok = false;
  for (int it = 0; it < kMaxPolar; ++it) {
    // cofactors C_ij = X_{i1 j1} X_{i2 j2} - X_{i1 j2} X_{i2 j1} and det = sum_j X_0j C_0j
    F3 C;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        fcfma(a, X.e[i1 * 3 + j1], X.e[i2 * 3 + j2]);
        fcfma(a, fneg(X.e[i1 * 3 + j2]), X.e[i2 * 3 + j1]);
        fnorm(a);
        C.e[i * 3 + j] = a;
      }
    float4 det = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 3; ++j) fcfma(det, X.e[j], C.e[j]);
    fnorm(det);
    const double2 dd = join_ff(det);
    const double dn = dd.x * dd.x + dd.y * dd.y;
    if (!(dn > 0.0) || !isfinite(dn)) break;
    const double inv_dn = 1.0 / dn;
    float nx = 0.f, nc = 0.f;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      nx = fmaf(X.e[e].x, X.e[e].x, fmaf(X.e[e].z, X.e[e].z, nx));
      nc = fmaf(C.e[e].x, C.e[e].x, fmaf(C.e[e].z, C.e[e].z, nc));
    }
    // Frobenius scaling gamma = sqrt(|X^-1|_F / |X|_F) = (|C|_F^2 / (|det|^2 |X|_F^2))^(1/4)
    const float gam = sqrtf(sqrtf(nc * (float)inv_dn / nx));
    const bool scale = fabsf(gam - 1.f) > 1e-3f;
    const float g1 = scale ? 0.5f * gam : 0.5f, g2 = scale ? 0.5f / gam : 0.5f;
    // X^{-+} = conj(C) det / |det|^2, elementwise; q = g2 det / |det|^2 (float-float)
    const float4 q = split_ff(make_double2((double)g2 * dd.x * inv_dn, (double)g2 * dd.y * inv_dn));
    const float4 g1c = make_float4(g1, 0.f, 0.f, 0.f);
    float diff = 0.f;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      float4 xn = make_float4(0.f, 0.f, 0.f, 0.f);
      fcfma(xn, g1c, X.e[e]);
      fcfma_ca(xn, C.e[e], q);
      fnorm(xn);
      const float dx = __fadd_rn(__fsub_rn(xn.x, X.e[e].x), __fsub_rn(xn.y, X.e[e].y));
      const float dy = __fadd_rn(__fsub_rn(xn.z, X.e[e].z), __fsub_rn(xn.w, X.e[e].w));
      diff = fmaf(dx, dx, fmaf(dy, dy, diff));
      X.e[e] = xn;
    }
    if (!isfinite(diff)) break;
    // unscaled and the step below 1e-9: Newton's quadratic convergence leaves an error ~1e-18
    if (!scale && diff < 1e-18f) {
      ok = true;
      break;
    }
  }
  if (!ok) {
    atomicExch(err, 1);
    return;
  }
#pragma unroll
  for (int e = 0; e < 9; ++e)
    *reinterpret_cast<ulonglong2*>(F + ((size_t)mu * 9 + e) * g.V + n) =
        make_ulonglong2(pk(X.e[e].x, X.e[e].z), pk(X.e[e].y, X.e[e].w));
}

// long_mu(n) = naik W_mu(n) W_mu(n+mu) W_mu(n+2mu), written in FP64 in host order [V][4][9]
__global__ void __launch_bounds__(3 * kSites) k_naik(Lat g, const C2* __restrict__ W, double naik,
                                                     double2* __restrict__ out) {
  const long n = (long)blockIdx.x * kSites + threadIdx.x, V = g.V;
  if (n >= V) return;
  const int i = threadIdx.y, mu = blockIdx.y;
  const Dir dmu = dir_of(g, n, mu);
  const C2* Wm = field(W, mu, V);
  R3 m, p;
  row_mul<PLAIN, true>(m, ld_row(Wm, V, n, i), Wm, V, n + dmu.off(1));
  row_mul<PLAIN, true>(p, m, Wm, V, n + dmu.off(2));
  double2* o = out + ((size_t)n * 4 + mu) * 9 + 3 * i;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double2 v = to_double(p.e[j]);
    o[j] = make_double2(naik * v.x, naik * v.y);
  }
}

int check_dims(const int dims[4], Lat* g) {
  if (!dims) return SQCG_ERR_INVALID_ARG;
  long V = 1;
  for (int d = 0; d < 4; ++d) {
    if (dims[d] < 4 || (dims[d] & 1)) return SQCG_ERR_INVALID_ARG;
    g->L[d] = dims[d];
    V *= dims[d];
  }
  if (V > (1L << 30)) return SQCG_ERR_INVALID_ARG;
  g->V = V;
  return SQCG_OK;
}

const sqcg_hisq_coeffs kDefaultCoeffs = {
    {1.0 / 8.0, 1.0 / 16.0, 1.0 / 64.0, 1.0 / 384.0, 0.0},
    {1.0, 1.0 / 16.0, 1.0 / 64.0, 1.0 / 384.0, -1.0 / 8.0},
    -1.0 / 24.0,
};

bool finite_level(const sqcg_smear_level& l) {
  return isfinite(l.one_link) && isfinite(l.three_staple) && isfinite(l.five_staple) && isfinite(l.seven_staple) &&
         isfinite(l.lepage);
}

// a coefficient as a float-float pair (hi = fl32(c), lo = fl32(c - hi)); zero stays (0, 0)
float2 ff_coeff(double c) {
  const float h = (float)c;
  return make_float2(h, (float)(c - (double)h));
}

// one smearing level: U (float-float fields) -> out (float-float fields, or FP64 host order when aos)
int smear_level(const Lat& g, const C2* U, C2* S, C2* Z, const sqcg_smear_level& c, int aos, void* out, cudaStream_t s) {
  const dim3 blk(kSites, 3);
  const unsigned gx = (unsigned)((g.V + kSites - 1) / kSites);
  const bool lepage = ff_coeff(c.lepage).x != 0.f;
  const bool staples57 = ff_coeff(c.five_staple).x != 0.f || ff_coeff(c.seven_staple).x != 0.f;
  const bool need_s = lepage || staples57 || ff_coeff(c.three_staple).x != 0.f;
  if (need_s) k_staple3<<<dim3(gx, 12), blk, 0, s>>>(g, U, S, lepage ? 1 : 0);
  if (lepage || staples57)
    k_staple57<<<dim3(gx, 12), blk, 0, s>>>(g, U, S, ff_coeff(c.five_staple), ff_coeff(c.seven_staple),
                                            ff_coeff(c.lepage), Z);
  const C2* Y = lepage ? S : staples57 ? Z : nullptr;
  k_smear_links<<<dim3(gx, 4), blk, 0, s>>>(g, U, S, Y, lepage ? 2 : 1, ff_coeff(c.one_link), ff_coeff(c.three_staple),
                                            aos, out);
  return cudaGetLastError() == cudaSuccess ? SQCG_OK : SQCG_ERR_CUDA;
}

}  // namespace

extern "C" size_t sqcg_hisq_workspace_bytes(const int dims[4]) {
  Lat g;
  if (check_dims(dims, &g) != SQCG_OK) return 0;
  // thin fields (4) + staples (kNumS) + Z (12) + level-1 result / projected links (4), then an error flag
  return (size_t)(4 + kNumS + 12 + 4) * 9 * g.V * sizeof(double2) + 256;
}

extern "C" int sqcg_hisq_smear(const int dims[4], const void* thin, void* fat, void* lng, const sqcg_hisq_coeffs* coeffs,
                               void* workspace, size_t workspace_bytes, void* stream) {
  Lat g;
  SQCG_TRY(check_dims(dims, &g));
  if (!thin || !fat || !lng || !workspace || fat == lng || thin == lng) return SQCG_ERR_INVALID_ARG;
  if ((((uintptr_t)thin) | ((uintptr_t)fat) | ((uintptr_t)lng) | ((uintptr_t)workspace)) & 15)
    return SQCG_ERR_INVALID_ARG;
  if (workspace_bytes < sqcg_hisq_workspace_bytes(dims)) return SQCG_ERR_INVALID_ARG;
  const sqcg_hisq_coeffs& c = coeffs ? *coeffs : kDefaultCoeffs;
  if (!finite_level(c.level1) || !finite_level(c.level2) || !isfinite(c.naik)) return SQCG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t nf = 9 * (size_t)g.V;
  C2* U = (C2*)workspace;  // float-float fields, 16 bytes per complex element
  C2* S = U + 4 * nf;
  C2* Z = S + kNumS * nf;
  C2* W = Z + 12 * nf;
  int* err = (int*)(W + 4 * nf);
  const unsigned gx = (unsigned)((g.V + kThreads - 1) / kThreads);
  SQCG_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  k_links_to_fields<<<dim3(gx, 4), kThreads, 0, s>>>(g, (const double2*)thin, U);
  SQCG_CUDA_TRY(cudaGetLastError());
  SQCG_TRY(smear_level(g, U, S, Z, c.level1, 0, W, s));
  k_u3_project<<<dim3(gx, 4), kThreads, 0, s>>>(g, W, err);
  SQCG_CUDA_TRY(cudaGetLastError());
  SQCG_TRY(smear_level(g, W, S, Z, c.level2, 1, fat, s));
  k_naik<<<dim3((unsigned)((g.V + kSites - 1) / kSites), 4), dim3(kSites, 3), 0, s>>>(g, W, c.naik, (double2*)lng);
  SQCG_CUDA_TRY(cudaGetLastError());
  int h_err = 0;
  SQCG_CUDA_TRY(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  SQCG_CUDA_TRY(cudaStreamSynchronize(s));
  return h_err ? SQCG_ERR_BREAKDOWN : SQCG_OK;
}

extern "C" int sqcg_hisq_load_links(sqcg_ctx* ctx, const double* thin, const sqcg_hisq_coeffs* coeffs, int opts,
                                    double* fat_out, double* lng_out) {
  if (!ctx || !thin) return SQCG_ERR_INVALID_ARG;
  if (ctx->flags & SQCG_PHASES_FOLDED) return SQCG_ERR_INVALID_ARG;  // the smearing takes unphased thin links
  if (opts & ~(SQCG_RECON12_LONG | SQCG_EIGHT_WAY)) return SQCG_ERR_INVALID_ARG;
  const size_t V = 2 * (size_t)ctx->g.Vh;
  const size_t bytes = V * 4 * 9 * sizeof(double2);
  const size_t wsb = sqcg_hisq_workspace_bytes(ctx->L);
  cudaStream_t s = ctx->stream;
  void *fat = nullptr, *lng = nullptr, *ws = nullptr;
  if (cudaMalloc(&fat, bytes) != cudaSuccess || cudaMalloc(&lng, bytes) != cudaSuccess ||
      cudaMalloc(&ws, wsb) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(fat); cudaFree(lng); cudaFree(ws);
    return SQCG_ERR_NO_MEMORY;
  }
  int rc = SQCG_OK;
  do {
    // the thin links are staged in the fat output buffer: the first kernel consumes them
    if (cudaMemcpyAsync(fat, thin, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) { rc = SQCG_ERR_CUDA; break; }
    if ((rc = sqcg_hisq_smear(ctx->L, fat, fat, lng, coeffs, ws, wsb, s)) != SQCG_OK) break;
    cudaFree(ws);
    ws = nullptr;
    if (fat_out && cudaMemcpyAsync(fat_out, fat, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) { rc = SQCG_ERR_CUDA; break; }
    if (lng_out && cudaMemcpyAsync(lng_out, lng, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) { rc = SQCG_ERR_CUDA; break; }
    if (cudaStreamSynchronize(s) != cudaSuccess) { rc = SQCG_ERR_CUDA; break; }
    rc = layout_load_links_device(ctx, (const double*)fat, (const double*)lng, opts);
  } while (0);
  if (rc == SQCG_ERR_CUDA) sqcg_set_last_cuda_error(cudaGetLastError(), "hisq_load_links", __FILE__, __LINE__);
  cudaStreamSynchronize(s);
  cudaFree(fat);
  cudaFree(lng);
  cudaFree(ws);
  return rc;
}
