// Persistent single-reduction mixed-precision CG: the whole Krylov loop between two reliable updates
// in one cooperative kernel, one resident grid that stays on the GPU from one reliable update to the
// next (arXiv:1611.00728 Sec. 4: the CG of the staggered normal equations, with the Dslash as its
// kernel).
//
// Each iteration is the single-reduction step of the graph-launched loop (cg.cu), in phases separated by
// grid-wide barriers instead of kernel boundaries. A block (one a SM) owns every gridDim.x-th group of 32
// sites of each parity:
//   U  (from the second step of a launch on) the previous step's vector update on its even groups,
//      p = r + beta p, q = s + beta q, xh += alpha p, r -= alpha q, and <r_new, q>
//   A  tmp = D_oe r on its odd groups
//   B  s = sigma r - D_eo tmp, with <r,s>, |r|^2 (and <r,q> right after a reliable update); the block posts
//      its sums
//   C  every block adds the posted sums in index order and runs the scalar step (convergence, reliable-
//      update trigger, alpha, beta) on its own copy of the solver state in shared memory: the sums
//      and the step are the same instructions on the same data in every block, so every copy is
//      identical and no broadcast is needed.
// FUSE: U and A run without a barrier between them; each neighbour's r_new is formed on the fly from the
// previous r, s and q with the same two FMAs its owner uses (so the values agree bit for bit), and r and q
// alternate between two buffers by step, so no block overwrites what another still reads. Without FUSE
// everything is updated in place and a third barrier follows U.
//
// What bounds it, and what the layout answers (one step at 8^4 took 23.9 us in the form before this one: one
// thread a site, a block per 128 sites; cycles of that step in brackets):
//  * a thread's chain of 16 hops, each waiting for L2 (2 x 7000): a group goes to SPLIT warps that share its
//    hops and meet in shared memory. Neighbour indices and, of few groups, as many of their links as fit are
//    kept in shared memory from the launch on, the 12-real rows already rebuilt. (2 x 1500 now)
//  * the grid barriers (2 x 4000): one counter that only grows, arrived at with a release and polled with an
//    acquire, by one block a SM. A tagged-slot barrier in which every block polled every other's sums took 8000.
//  * the sums (3300): three warps add one sum each, one round of loads for the 152 blocks (1250)
//  * the scalar step in FP64 (2500; an FP64 operation holds its scheduler for 64 cycles): in float-float, with
//    the FP64 state and the reciprocal of gamma formed by other warps at the next barrier (step_ff; 500)
// A step takes 5.6 us at 8^4, 7.9 on 10x12x14x16 and 13.0 at 16^4; an iteration of a solve, launches and reliable
// updates with it, 7.9 (22.1), 9.8 (22.4), 15.6 (25.1) and at 20^4 29.5 (36.7; full links 34.7 / 43.8).
//
// The kernel returns when the step asks for a reliable update or the solve is done, with r and q
// in the context's buffers; block 0 writes its state copy back. The true-residual pass (float-float or FP64
// Dslash pair) follows on the stream, gated by that state, then the kernel again, which starts with the
// three-sum phase B (cg.cu).
//
// Every phase reads the vectors other blocks wrote in the phase before through coherent loads (not
// the read-only path); the links are read-only and keep it. A wait at a barrier ends after kBarrierSpins
// polls: the block records the time-out, the grid leaves the loop and the state reports SQCG_ERR_CUDA. The
// launch is cooperative, so the runtime refuses a grid that cannot be resident at once instead of starting it.
#include <stdlib.h>
#include <string.h>

#include "dslash_core.cuh"

namespace {

using namespace dcore;

// a wait gives up after this many polls (each a round trip to L2, 0.4 us): well over a thousand times the
// longest phase a barrier waits for in a solve
constexpr unsigned kBarrierSpins = 1u << 20;

struct PArgs {
  DArgs<float> d1;  // tmp = D_oe r  (output parity 1, in = r, out = tmp)
  DArgs<float> d2;  // s = sigma r - D_eo tmp  (output parity 0, in = tmp, out = s)
  float2* r;   // r and q (with FUSE of even steps; the context's buffers, in and out)
  float2* r1;  // FUSE: ... and of odd steps
  float2* s;
  float2* p;
  float2* q;
  float2* q1;
  float2* xh;
  float2* tmp;
  int Vh, ngroups;
  SolverState* st;
  float2* slots;      // [3][G] the blocks' totals of the step's sums <r,s>, <r,q>, |r|^2 (float-float)
  unsigned* bar;      // [0] arrivals, [1] time-out flag; zero at launch
  int max_mine;       // groups of the block that has most; 0: too many to keep their neighbour indices
  int ncached;        // hop links a block keeps in shared memory
  int max_iter;     // bound on the state's iteration count (the solver state ends the loop sooner)
  unsigned arrivals;  // blocks a barrier waits for: the grid (one more only in the time-out test)
};

__device__ __forceinline__ void warp_sum_ffs(float2& v) {  // total in lane 0
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = ffs_add(v, make_float2(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o)));
}

// Grid-wide barrier number n (from 1): one counter that only grows. While thread 0 waits, the other
// warps run idle(). False when a wait timed out (here or elsewhere).
template <typename F>
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned n, unsigned arrivals, const F& idle) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const unsigned target = n * arrivals;  // the counter may wrap: compare differences
    int good = 1;
    for (unsigned spins = 0;; ++spins) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if (spins > kBarrierSpins || ((spins & 63u) == 63u && *(volatile unsigned*)(bar + 1) != 0u)) {
        atomicExch(bar + 1, 1u);
        good = 0;
        break;
      }
    }
    ok = good;
  } else if (threadIdx.x >= 32) {
    idle();
  }
  __syncthreads();
  return ok != 0;
}

// The scalar step of a plain continuing iteration (sr_step, solver_device.cuh) in float-float on the FP32
// pipe. An FP64 operation holds its scheduler for 64 cycles on this GPU whatever the lanes in it, and the
// whole grid waits for this chain: some 30 of them took 2900 cycles, this takes 500. Only what the next phase
// needs comes out of it, alpha and beta in FP32; the FP64 state follows while the grid waits at the
// next barrier, from the same sums. Errors of 84 solves (4x6x8x10 to 20^4, to 1e-11) against 64 bits: 1.0005 +- 0.0002
// of the graph loop's, whose step is sr_step. False where sr_step itself has to run: a reliable update or
// the end of the solve, or numbers outside the range in which the float-float chain is safe.
struct StepInputs {  // formed at the barrier before
  float2 inv;   // 1 / gamma_{k-1}
  float2 pAp;   // <p_{k-1}, q_{k-1}>
  float2 stop;  // gamma at which the solve ends ...
  float2 update;  // ... and below which a reliable update is due
};
__device__ __forceinline__ float2 ffs_split(double v) {
  const float h = (float)v;
  return make_float2(h, (float)(v - (double)h));
}
__device__ __forceinline__ float2 ffs_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.y, b.x, fmaf(a.x, b.y, fmaf(a.x, b.x, -p)));
  const float h = __fadd_rn(p, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, p)));
}
__device__ __forceinline__ bool ffs_less(float2 a, float2 b) { return a.x < b.x || (a.x == b.x && a.y < b.y); }
__device__ __forceinline__ bool step_ff(const StepInputs& in, bool first, float2 d, float2 c, float2 g, float& alpha,
                                        float& beta) {
  constexpr float kLow = 1e-30f, kHigh = 1e30f;
  if (!(g.x > kLow && g.x < kHigh) || !(first || (in.inv.x < kHigh && in.pAp.x < kHigh))) return false;
  if (!ffs_less(in.stop, g) || ffs_less(g, in.update)) return false;
  float2 b = make_float2(0.f, 0.f), P = d;
  if (!first) {
    b = ffs_mul(g, in.inv);
    P = ffs_add(d, ffs_mul(b, ffs_add(make_float2(2.f * c.x, 2.f * c.y), ffs_mul(b, in.pAp))));
  }
  if (!(P.x > kLow && P.x < kHigh)) return false;
  const float r = __frcp_rn(P.x), q = __fmul_rn(g.x, r);
  alpha = fmaf(__fadd_rn(fmaf(-q, P.y, fmaf(-q, P.x, g.x)), g.y), r, q);
  beta = b.x;
  return true;
}

// r_new = r - alpha (s + beta q) at a neighbour, with the FMAs of the vector update
struct UpdatedIn {
  const float2* r;
  const float2* s;
  const float2* q;
  int Vh;
  float alpha, beta;
  __device__ __forceinline__ void operator()(float2 (&v)[3], int idx) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t k = (size_t)c * Vh + idx;
      const float2 rc = r[k], sc = s[k], qc = q[k];
      const float qx = fmaf(beta, qc.x, sc.x), qy = fmaf(beta, qc.y, sc.y);
      v[c] = make_float2(fmaf(-alpha, qx, rc.x), fmaf(-alpha, qy, rc.y));
    }
  }
};

constexpr size_t kMaxSmem = 206 * 1024;    // dynamic shared memory of a launch; k_sr_persistent's own comes on top
constexpr size_t kBlockSmem = 227 * 1024;  // what a block can have
constexpr int kLinkFloats = 9 * 32;  // float2 of one hop's links of a 32-site group in shared memory

// Hop h of site i of group t (parity par's output): index of the neighbour, with the sign bit set where the
// scale of a 12-real long link is negative.
template <bool RECON, bool EIGHT>
__device__ __forceinline__ int hop_index(const DArgs<float>& a, int i, int h) {
  const Geom& g = a.g;
  const int xh = i % g.Lxh;
  int r = i / g.Lxh;
  const int y = r % g.Ly;
  r /= g.Ly;
  const int z = r % g.Lz;
  const int t = r / g.Lz;
  const int x = 2 * xh + ((y + z + t + a.par) & 1);
  const int mu = h >> 2, lng = (h >> 1) & 1, bwd = h & 1, d = lng ? 3 : 1;
  int nb;
  if (mu == 0) {
    int xn = bwd ? x - d : x + d;
    if (xn >= g.Lx) xn -= g.Lx;
    if (xn < 0) xn += g.Lx;
    nb = i - xh + (xn >> 1);
  } else {
    const int cmu = (mu == 1) ? y : (mu == 2) ? z : t;
    const int Lmu = (mu == 1) ? g.Ly : (mu == 2) ? g.Lz : g.Lt;
    const int smu = (mu == 1) ? g.sy : (mu == 2) ? g.sz : g.st;
    nb = bwd ? i - d * smu : i + d * smu;
    if (!bwd && cmu + d >= Lmu) nb -= Lmu * smu;
    if (bwd && cmu - d < 0) nb += Lmu * smu;
  }
  if (RECON && lng) {  // eta_mu(n), the boundary sign of the hop, and the sign of -L^+ (see dslash_site_in)
    const int e = (mu == 0) ? 0 : (mu == 1) ? x : (mu == 2) ? x + y : x + y + z;
    bool neg = e & 1;
    if (mu == 3 && g.apbc && (bwd ? t < 3 : t + 3 >= g.Lt)) neg = !neg;
    if (EIGHT && bwd) neg = !neg;
    if (neg) nb |= (int)0x80000000;
  }
  return nb;
}

// the link of hop h at site i (index word e of hop_index), third row rebuilt
template <bool RECON, bool EIGHT>
__device__ __forceinline__ void hop_link(const DArgs<float>& a, int i, int h, int e, float2 (&U)[9]) {
  const int mu = h >> 2, lng = (h >> 1) & 1, bwd = h & 1, Vh = a.g.Vh;
  const int at = EIGHT || !bwd ? i : e & 0x7fffffff;
  if (!lng) {
    const float2* base = !bwd ? a.fat_p : EIGHT ? a.fatb_p : a.fat_q;
    load_link<float, float2, false>(U, base + (size_t)mu * 9 * Vh, Vh, at, 1.f);
  } else {
    const float2* base = !bwd ? a.lng_p : EIGHT ? a.lngb_p : a.lng_q;
    load_link<float, float2, RECON>(U, base + (size_t)mu * a.nl * Vh, Vh, at, e < 0 ? -a.inv_s0 : a.inv_s0);
  }
}

template <bool RECON, bool EIGHT, int SPLIT, int NW, bool FUSE>
__global__ void __launch_bounds__(32 * NW, 1) k_sr_persistent(PArgs a) {
  constexpr int NG = NW / SPLIT;  // groups in hand at once
  constexpr int NH = 16 / SPLIT;  // hops of a warp
  constexpr int PT = 32 * NW;
  static_assert(3 * NG < NW, "a warp per group and colour in the epilogue");
  // without this no block is resident, and the solve goes to the graph loop, correct but slower
  static_assert(kMaxSmem + sizeof(SolverState) + (9 * NG * 32 + NW) * sizeof(float2) + 128 <= kBlockSmem,
                "shared memory of a block: the state, part, wcross and a few words, beside kMaxSmem");
  // dynamic shared memory: the hops' partial sums [2][NW][3][32] (alternating by round: one barrier a
  // round), the neighbour indices [2][max_mine][16][32], then the cached links
  extern __shared__ float2 smx[];
  __shared__ SolverState ss;
  __shared__ float2 part[3][3 * NG][32], wcross[NW];  // the epilogue lanes' sums, the warps' cross terms
  __shared__ float2 total[3];  // <r,s>, <r,q>, |r|^2
  __shared__ StepInputs in;
  __shared__ float sc[3];  // alpha, beta, sigma of the step in FP32
  __shared__ double inv_prev[2];  // by step: step_state of one step and the next step's division overlap
  __shared__ int pending;         // the FP64 state does not hold the last step yet
  typedef unsigned long long W;
  constexpr int kWords = sizeof(SolverState) / sizeof(W);
  static_assert(sizeof(SolverState) % sizeof(W) == 0, "state copied as 8-byte words");
  for (int k = threadIdx.x; k < kWords; k += PT) reinterpret_cast<W*>(&ss)[k] = reinterpret_cast<const W*>(a.st)[k];
  const int G = gridDim.x, Vh = a.Vh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mine = (a.ngroups - 1 - (int)blockIdx.x) / G + 1;  // this block's groups (G <= ngroups)
  __syncthreads();
  if (threadIdx.x == 0) {
    ss.use_if = 0;
    sc[2] = (float)ss.sigma;
    pending = 0;
    in.stop = ffs_split(ss.stop_rr);
  }
  if (ss.done || ss.need_update) return;  // uniform over the grid
  int* nbr = reinterpret_cast<int*>(smx + 2 * NW * 96);
  float2* links = reinterpret_cast<float2*>(nbr + 2 * a.max_mine * 512);
  // the slot of hop h of group t and parity par among the cached links, in an order that spreads the
  // cached hops over the warps of a group; cached where it is below a.ncached
  auto link_slot = [&](int par, int t, int h) { return (((h % NH) * SPLIT + h / NH) * 2 + par) * mine + t; };
  for (int task = warp; task < 2 * 16 * mine && a.max_mine; task += NW) {
    const int h = task & 15, t = (task >> 4) % mine, par = (task >> 4) / mine;
    const DArgs<float>& da = par ? a.d1 : a.d2;
    const int i = ((int)blockIdx.x + t * G) * 32 + lane;
    if (i < Vh) {
      const int e = hop_index<RECON, EIGHT>(da, i, h);
      nbr[((par * mine + t) * 16 + h) * 32 + lane] = e;
      const int slot = link_slot(par, t, h);
      if (slot < a.ncached) {
        float2 U[9];
        hop_link<RECON, EIGHT>(da, i, h, e, U);
#pragma unroll
        for (int k = 0; k < 9; ++k) links[slot * kLinkFloats + k * 32 + lane] = U[k];
      }
    }
  }
  __syncthreads();
  bool timed_out = false;
  unsigned nbar = 0;
  int round = 0;
  // D on this block's groups of parity par; out(c, i, d) takes colour c of site i, in one warp per group and colour
  auto dslash_groups = [&](int par, const DArgs<float>& da, const auto& in_at, auto&& out) {
    for (int t0 = 0; t0 < mine; t0 += NG, ++round) {
      float2* buf = smx + (round & 1) * NW * 96;
      {
        const int t = t0 + warp / SPLIT, part = warp % SPLIT;
        const int i = ((int)blockIdx.x + t * G) * 32 + lane;
        if (t < mine && i < Vh) {
          float2 acc[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) acc[c] = make_float2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < NH; ++j) {
            const int h = part * NH + j;
            const int e = a.max_mine ? nbr[((par * mine + t) * 16 + h) * 32 + lane] : hop_index<RECON, EIGHT>(da, i, h);
            float2 U[9], v[3];
            in_at(v, e & 0x7fffffff);
            const int slot = link_slot(par, t, h);
            if (slot < a.ncached) {
#pragma unroll
              for (int k = 0; k < 9; ++k) U[k] = links[slot * kLinkFloats + k * 32 + lane];
            } else {
              hop_link<RECON, EIGHT>(da, i, h, e, U);
            }
            if (EIGHT || !(h & 1)) acc_mv<float>(acc, U, v);
            else sub_mdv<float>(acc, U, v);
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) buf[(warp * 3 + c) * 32 + lane] = acc[c];
        }
      }
      __syncthreads();
      if (warp < 3 * NG) {
        const int sub = warp / 3, c = warp % 3;
        const int i = ((int)blockIdx.x + (t0 + sub) * G) * 32 + lane;
        if (t0 + sub < mine && i < Vh) {
          float2 d = buf[(sub * SPLIT * 3 + c) * 32 + lane];
#pragma unroll
          for (int w = 1; w < SPLIT; ++w) {
            const float2 u = buf[((sub * SPLIT + w) * 3 + c) * 32 + lane];
            d.x += u.x;
            d.y += u.y;
          }
          out(c, i, d);
        }
      }
    }
  };
  int n = 0;
  int cur = 0;  // buffer of the current r and q
  const float2 z = make_float2(0.f, 0.f);
  const int steps = a.max_iter - ss.iter;
  for (; n < steps; ++n) {
    const int cb = FUSE ? n & 1 : 0;  // this step's buffers
    float2* rn = cb ? a.r1 : a.r;
    float2* qn = cb ? a.q1 : a.q;
    const float2* ro = !FUSE ? a.r : cb ? a.r : a.r1;
    const float2* qo = !FUSE ? a.q : cb ? a.q : a.q1;
    const float alpha = sc[0], beta = sc[1], sig = sc[2];
    const bool after = ss.after_update != 0;
    float2 cross = z;
    // U: the previous step's update, a warp (but the first) per group and colour, with <r_new, q>
    if (n > 0 && warp > 0)
      for (int task = warp - 1; task < 3 * mine; task += NW - 1) {
        const int i = ((int)blockIdx.x + (task / 3) * G) * 32 + lane;
        if (i < Vh) {
          const size_t k = (size_t)(task % 3) * Vh + i;
          float2 rc = ro[k], pc = a.p[k], qc = qo[k], xc = a.xh[k];
          const float2 sv = a.s[k];
          pc.x = fmaf(beta, pc.x, rc.x);
          pc.y = fmaf(beta, pc.y, rc.y);
          qc.x = fmaf(beta, qc.x, sv.x);
          qc.y = fmaf(beta, qc.y, sv.y);
          xc.x = fmaf(alpha, pc.x, xc.x);
          xc.y = fmaf(alpha, pc.y, xc.y);
          rc.x = fmaf(-alpha, qc.x, rc.x);
          rc.y = fmaf(-alpha, qc.y, rc.y);
          a.p[k] = pc;
          qn[k] = qc;
          a.xh[k] = xc;
          rn[k] = rc;
          cross = ffs_add(cross, make_float2(fmaf(rc.x, qc.x, rc.y * qc.y), 0.f));
        }
      }
    if (!FUSE && n > 0 && !grid_barrier(a.bar, ++nbar, a.arrivals, [] {})) { timed_out = true; break; }
    // A: tmp = D_oe r
    auto put = [&](int c, int i, float2 d) { a.tmp[(size_t)c * Vh + i] = d; };
    if (FUSE && n > 0)
      dslash_groups(1, a.d1, UpdatedIn{ro, a.s, qo, Vh, alpha, beta}, put);
    else
      dslash_groups(1, a.d1, PlainIn<float2, false>{rn, Vh}, put);
    cur = cb;
    // while the first warp waits: the warps' cross terms, the FP64 state of the step before, and what the
    // next scalar step takes from it
    if (!grid_barrier(a.bar, ++nbar, a.arrivals, [&] {
          warp_sum_ffs(cross);
          if (lane == 0) wcross[warp] = cross;
          if (threadIdx.x == 32) {
            if (pending) {
              const double b = ss.iter == 1 ? 0.0 : ffs_value(total[2]) * inv_prev[(n - 1) & 1];
              ss.beta = b;
              ss.pAp = fma(b, fma(b, ss.pAp, 2.0 * ffs_value(total[1])), ffs_value(total[0]));
            }
            in.pAp = ffs_split(ss.pAp);
          }
          if (threadIdx.x == 64) {
            if (pending) {
              const double g = ffs_value(total[2]);
              ss.rr_prev = ss.rr;
              ss.rr = g;
              if (g > ss.rr_max) ss.rr_max = g;
            }
            const double inv = 1.0 / (after ? ss.rr_prev : ss.rr);
            inv_prev[n & 1] = inv;
            in.inv = ffs_split(inv);
            in.update = ffs_split(ss.delta2 * ss.rr_max);
          }
        })) {
      timed_out = true;
      break;
    }
    // B: s = sigma r - D_eo tmp with <r,s>, |r|^2 and, after a reliable update, <r,q>
    float2 v[3] = {z, z, z};
    dslash_groups(0, a.d2, PlainIn<float2, false>{a.tmp, Vh}, [&](int c, int i, float2 d) {
      const size_t k = (size_t)c * Vh + i;
      const float2 rc = rn[k];
      const float2 o = make_float2(sig * rc.x - d.x, sig * rc.y - d.y);
      a.s[k] = o;
      v[0] = ffs_add(v[0], make_float2(fmaf(rc.x, o.x, rc.y * o.y), 0.f));
      v[2] = ffs_add(v[2], make_float2(fmaf(rc.x, rc.x, rc.y * rc.y), 0.f));
      if (after) {
        const float2 qc = qn[k];
        v[1] = ffs_add(v[1], make_float2(fmaf(rc.x, qc.x, rc.y * qc.y), 0.f));
      }
    });
    if (warp < 3 * NG)
#pragma unroll
      for (int k = 0; k < 3; ++k) part[k][warp][lane] = v[k];
    __syncthreads();
    if (warp < 3) {  // warp k: the block's sum k
      float2 t = z;
      if (warp == 1 && !after) {
        if (lane > 0 && lane < NW) t = wcross[lane];
      } else {
        t = part[warp][0][lane];
#pragma unroll
        for (int w = 1; w < 3 * NG; ++w) t = ffs_add(t, part[warp][w][lane]);
      }
      warp_sum_ffs(t);
      if (lane == 0) a.slots[warp * G + blockIdx.x] = t;
    }
    if (!grid_barrier(a.bar, ++nbar, a.arrivals, [] {})) { timed_out = true; break; }
    // C: the step's sums, in the same order in every block, and the scalar step on the block's copy
    if (warp < 3) {
      constexpr int U = 5;  // slots of a lane in flight: one round for the 152 blocks of a full grid
      float2 t = z;
      for (int j0 = lane; j0 < G; j0 += 32 * U) {
        float2 w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = j0 + 32 * u < G ? a.slots[warp * G + j0 + 32 * u] : z;
#pragma unroll
        for (int u = 0; u < U; ++u) t = ffs_add(t, w[u]);
      }
      warp_sum_ffs(t);
      if (lane == 0) total[warp] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float al, be;
      if (!after && ss.iter < ss.max_iter && ss.iter - ss.iter_last_update < ss.update_interval &&
          step_ff(in, ss.iter == 0, total[0], total[1], total[2], al, be)) {
        sc[0] = al;
        sc[1] = be;
        ss.iter += 1;
        pending = 1;
      } else {
        sr_step(&ss, ffs_value(total[0]), ffs_value(total[1]), ffs_value(total[2]));
        sc[0] = (float)ss.alpha;
        sc[1] = (float)ss.beta;
        pending = 0;
      }
    }
    __syncthreads();
    if (ss.done || ss.need_update) break;  // the same decision in every block
  }
  // r and q back into the context's buffers (each block copies the even groups it wrote; nothing reads
  // them any more in this launch)
  if (FUSE && cur == 1) {
    for (int task = warp; task < 3 * mine; task += NW) {
      const int i = ((int)blockIdx.x + (task / 3) * G) * 32 + lane;
      if (i < Vh) {
        const size_t k = (size_t)(task % 3) * Vh + i;
        a.r[k] = a.r1[k];
        a.q[k] = a.q1[k];
      }
    }
  }
  if (blockIdx.x != 0) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    if (timed_out) {
      ss.status = SQCG_ERR_CUDA;
      ss.done = 1;
      ss.need_update = 0;
    } else if (!ss.done && !ss.need_update) {
      ss.status = SQCG_ERR_NOT_CONVERGED;
      ss.done = 1;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kWords; k += PT) reinterpret_cast<W*>(a.st)[k] = reinterpret_cast<const W*>(&ss)[k];
}

struct PKernel {
  void* fn;
  int threads;
  size_t smem_fixed;  // partial sums; the indices and links follow
};

template <bool RECON, bool EIGHT, int SPLIT, int NW, bool FUSE>
PKernel kernel_of() {
  return {reinterpret_cast<void*>(k_sr_persistent<RECON, EIGHT, SPLIT, NW, FUSE>), 32 * NW,
          (size_t)2 * NW * 96 * sizeof(float2)};
}

template <int SPLIT, int NW, bool FUSE>
PKernel kernel_for(const sqcg_ctx* ctx) {
  if (ctx->eightway) return ctx->recon ? kernel_of<true, true, SPLIT, NW, FUSE>() : kernel_of<false, true, SPLIT, NW, FUSE>();
  return ctx->recon ? kernel_of<true, false, SPLIT, NW, FUSE>() : kernel_of<false, false, SPLIT, NW, FUSE>();
}

// The kernel for the context's link form and lattice, by the 32-site groups of the block that has most. Measured, us an
// iteration of a solve (12-real, to 1e-11), SPLIT x warps: fused 16x16 / fused 8x24 / 8x32 / 4x24:
//    1 group  (8^4)           7.9 /  8.7 / 10.3 / 11.1     11 groups (18^4)         28.2 / 22.7 / 21.9 / 21.2
//    2 groups (8^3x32)        7.5 /  7.4 /  9.0 /  9.7     12 groups (18^3x20)      28.7 / 23.6 / 22.4 / 21.6
//    3 groups (10x12x14x16)  10.6 /  9.8 / 10.9 / 11.3     14 groups (16x18x20x22)  30.4 / 25.7 / 24.2 / 24.5
//    4 groups (14^4)         13.0 / 12.8 / 12.5 / 12.6     15 groups (18x18x20x22)  41.7 / 29.9 / 26.1 / 26.5
//    5 groups (12x14x16x18)  14.5 / 13.4 / 14.2 / 13.1     16 groups (16x20x22x22)  44.0 / 33.1 / 27.1 / 27.9
//    6 groups (14^3x18)      16.3 / 14.3 / 14.5 / 13.5     17 groups (20^4)         50.5 / 34.8 / 30.8 / 29.4
//    7 groups (16^4)         17.9 / 16.6 / 15.6 / 17.3     18 groups (18x20x22x22)  57.4 / 38.6 / 32.9 / 31.9
//    8 groups (16^3x18)      19.6 / 17.5 / 16.7 / 18.3     19 groups (20^3x22)      60.9 / 43.7 / 34.1 / 37.9
//    9 groups (16x16x18x18)  21.7 / 18.5 / 19.1 / 18.9     20 groups (20x20x22x22)  70.3 / 49.1 / 37.4 / 42.5
//   10 groups (16x18x16x20)  23.4 / 21.0 / 20.0 / 19.3     22 groups (22x22x20x22)  80.7 / 58.1 / 48.1 / 48.9
// Forming r_new on the fly trades a barrier for three times the gathers, which pays only while a block has few groups.
// Above, a block takes four groups a round with 8x32 and six with 4x24, whose rounds take about half as long again:
// 4x24 where 8x32 needs one and a half times the rounds.
PKernel persistent_kernel(const sqcg_ctx* ctx) {
  const int mine = (grid_for(ctx->g.Vh, 32) + ctx->nsm - 1) / ctx->nsm;
  if (mine <= 1) return kernel_for<16, 16, true>(ctx);
  if (mine <= 3) return kernel_for<8, 24, true>(ctx);
  const int rounds32 = (mine + 3) / 4, rounds24 = (mine + 5) / 6;
  return 2 * rounds32 >= 3 * rounds24 ? kernel_for<4, 24, false>(ctx) : kernel_for<8, 32, false>(ctx);
}

DArgs<float> dargs(const sqcg_ctx* ctx, int par, const float2* in, float2* out) {
  DArgs<float> a = {};
  const size_t Vh = ctx->g.Vh;
  const int p = par, q = 1 - par;
  const int nl = ctx->recon ? 6 : 9;
  const float2* fat = reinterpret_cast<const float2*>(ctx->fat32);
  const float2* lng = reinterpret_cast<const float2*>(ctx->lng32);
  a.g = ctx->g;
  a.par = par;
  a.fat_p = fat + (size_t)p * 4 * 9 * Vh;
  a.fat_q = fat + (size_t)q * 4 * 9 * Vh;
  a.lng_p = lng + (size_t)p * 4 * nl * Vh;
  a.lng_q = lng + (size_t)q * 4 * nl * Vh;
  a.fatb_p = ctx->eightway ? reinterpret_cast<const float2*>(ctx->fatb32) + (size_t)p * 4 * 9 * Vh : nullptr;
  a.lngb_p = ctx->eightway ? reinterpret_cast<const float2*>(ctx->lngb32) + (size_t)p * 4 * nl * Vh : nullptr;
  a.nl = nl;
  a.inv_s0 = (float)(ctx->recon ? 1.0 / ctx->long_scale : 1.0);
  a.in = in;
  a.out = out;
  return a;
}

// Dynamic shared memory of a launch: the kernel's own, the neighbour indices of the fullest block's groups where
// they fit (*max_mine, else 0), and as many of their hop links (*ncached) as still do, where that is a sixth of them
// (an eighth of 8-way 12-real ones, which no other site reads): what a block does not take is L1, which serves the
// gathers. us an iteration with / without links in shared memory: 16^4 (7 groups a block, a quarter of them) 15.8 / 16.7,
// 16^3x18 (8) 16.7 / 17.3, 16x18x16x20 (10, 18%) 19.4 / 19.6, 18^4 (11, 16%) 21.7 / 21.2 (full 23.1 / 21.2; 8-way
// 12-real 28.1 / 30.3), 20^4 (17) 31.8 / 29.9 (full 43.2 / 35.5), 20^3x22 (19) 40.8 / 34.3 (full 54.9 / 42.4).
size_t smem_bytes(const PKernel& k, const sqcg_ctx* ctx, int* max_mine, int* ncached) {
  const size_t mine = (grid_for(ctx->g.Vh, 32) + ctx->nsm - 1) / ctx->nsm;
  const size_t base = k.smem_fixed + 2 * mine * 512 * sizeof(int), link = kLinkFloats * sizeof(float2);
  *max_mine = *ncached = 0;
  if (base > kMaxSmem) return k.smem_fixed;
  const size_t fit = (kMaxSmem - base) / link, all = 32 * mine;
  size_t n = fit < all ? fit : all;
  if ((ctx->eightway && ctx->recon ? 8 : 6) * n < all) n = 0;
  *max_mine = (int)mine;
  *ncached = (int)n;
  return base + n * link;
}

// the blocks' totals, then the barrier words
size_t pers_sync_bytes(const sqcg_ctx* ctx) { return 3 * (size_t)ctx->nsm * sizeof(float2) + 2 * sizeof(unsigned); }

}  // namespace

// Grid of the persistent loop for the context's link form (0: not available): one resident block a SM,
// never more blocks than 32-site groups. Allocates the kernel's partials and barrier words on first use.
int persistent_grid(sqcg_ctx* ctx) {
  if (ctx->pers_grid < 0) return 0;
  const PKernel k = persistent_kernel(ctx);
  if (ctx->pers_grid > 0 && ctx->pers_fn == k.fn) return ctx->pers_grid;
  int dev = 0, coop = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
      cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, kMaxSmem) != cudaSuccess) {
    cudaGetLastError();
    ctx->pers_grid = -1;
    return 0;
  }
  if (!coop || per_sm < 1) {
    ctx->pers_grid = -1;
    return 0;
  }
  if (!ctx->pers_sync) {
    const size_t nv = (size_t)3 * ctx->g.Vh;
    if (cudaMalloc(&ctx->pers_sync, pers_sync_bytes(ctx)) != cudaSuccess ||
        cudaMalloc(&ctx->pers_rq, 2 * nv * sizeof(float2)) != cudaSuccess) {
      cudaGetLastError();
      cudaFree(ctx->pers_sync);
      cudaFree(ctx->pers_rq);
      ctx->pers_sync = nullptr;
      ctx->pers_rq = nullptr;
      ctx->pers_grid = -1;
      return 0;
    }
  }
  const int ngroups = grid_for(ctx->g.Vh, 32);
  ctx->pers_fn = k.fn;
  ctx->pers_grid = ngroups < ctx->nsm ? ngroups : ctx->nsm;  // one block a SM
  return ctx->pers_grid;
}

// One launch of the persistent loop on the solver workspace (r32, Ap32 as s, p32, q32, xh32, tmp32).
int launch_sr_persistent(sqcg_ctx* ctx, int max_iter, cudaStream_t s) {
  const int G = persistent_grid(ctx);
  if (G <= 0) return SQCG_ERR_INVALID_ARG;
  PArgs a = {};
  a.d1 = dargs(ctx, 1, ctx->r32, ctx->tmp32);
  a.d2 = dargs(ctx, 0, ctx->tmp32, ctx->Ap32);
  a.r = ctx->r32;
  a.r1 = ctx->pers_rq;
  a.s = ctx->Ap32;
  a.p = ctx->p32;
  a.q = ctx->q32;
  a.q1 = ctx->pers_rq + (size_t)3 * ctx->g.Vh;
  a.xh = ctx->xh32;
  a.tmp = ctx->tmp32;
  a.Vh = ctx->g.Vh;
  a.ngroups = grid_for(ctx->g.Vh, 32);
  a.st = ctx->st;
  a.slots = (float2*)ctx->pers_sync;
  a.bar = (unsigned*)(a.slots + 3 * (size_t)ctx->nsm);
  a.max_iter = max_iter;
  // SQCG_TEST_BARRIER_TIMEOUT=1 makes every barrier wait for one block more than the grid has, so each
  // wait runs out: the test of the bounded waits (the solve then returns SQCG_ERR_CUDA, nothing hangs)
  const char* t = getenv("SQCG_TEST_BARRIER_TIMEOUT");
  a.arrivals = (unsigned)G + ((t && strcmp(t, "1") == 0) ? 1u : 0u);
  SQCG_CUDA_TRY(cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), s));
  const PKernel k = persistent_kernel(ctx);
  const size_t smem = smem_bytes(k, ctx, &a.max_mine, &a.ncached);
  void* args[] = {&a};
  SQCG_CUDA_TRY(cudaLaunchCooperativeKernel(k.fn, dim3(G), dim3(k.threads), args, smem, s));
  return SQCG_OK;
}
