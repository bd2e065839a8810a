// Level CG with the level's vectors resident in shared memory, for one grid of up to a
// few hundred thousand nodes (the middle levels of the cascade, where a CG step is bound
// by latency, not by the FP64 pipe or HBM).
//
// A cooperative grid of G blocks; block b owns a box of BX x BY x BZ interior nodes and
// keeps in shared memory, for all steps of the level, x, p, s, w of its box and r of its
// box plus a one-node halo.  The recurrence is the single-reduction form of CG of
// Chronopoulos and Gear (1989), as in the cluster kernel:
//
//    p = r + beta p,  s = w + beta s,  x += alpha p,  r -= alpha s,
//    w = A r,  gamma = r.r,  delta = w.r   (one grid reduction for both),
//    beta' = gamma' / gamma,  alpha' = gamma' / (delta' - beta' gamma' / alpha);
//
// in exact arithmetic x and r are those of the standard recurrence (the smoother of
// Algorithm 1), and the loop stops on the same recursive residual r.r <= tol2.
//
// Halo exchange through global memory (L2): every step each block publishes the new r, s
// and w of its box into node arrays of the level (two copies by step parity), and the
// next step recomputes the new r on its halo from its neighbours' published r, w, s with
// the same fused operations as the owner (bit-identical).  So one step needs one grid-wide
// synchronisation, the reduction's: per-block sums, one arrival counter (release /
// acquire, bounded wait: EXCMG_ERR_TIMEOUT), then every block adds the G blocks' sums, so
// all blocks hold bit-identical scalars and take the same decisions.
//
// What bounds a step: the chain of its parts on the smallest levels, the FP64 pipe on the
// largest.  A float64 warp instruction takes the pipe 64 clocks whatever its lanes do, so
// the 19-point sums (fixed_point.cuh) and the reductions run on integers, and float64 is
// left with the vector updates, the two products and the scalars: 8.5 instructions per node
// and step instead of 25.  Measured per step, all in float64 and now: 16^3 cells 6.2 us, 4.5;
// 32^3 7.5, 5.2; 64^3 22.0, 11.2; 128 x 64 x 64 37.7, 19.8 (3.8, 4.7, 9.8, 18.0 with sums of fewer
// bits and no check of small values).  A field that falls off within its boxes has them in float64
// too: 40 steps from zero on 64^3 with u = exp(-100 x) 1.29 ms, 1.12 in float64 alone (a box that stays
// in float64 for 1, 3 or 7 steps after one: 1.23, 1.19, 1.17, and whole solves 0 to 4% slower).
// The blocks' sums are read by all warps (one or two per thread): read by one warp, ten per
// lane, they cost 1.5 us more.
#include <cuda_runtime.h>

#include <algorithm>

#include "excmg_internal.cuh"
#include "fixed_point.cuh"

namespace excmg {
namespace {

constexpr int kRsThreads = 256;
constexpr unsigned long long kRsSpinLimit = 1ull << 25;
constexpr int kRsHB = 6;  // halo nodes per thread whose loads are issued ahead

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ double rs_xor_sum(double v, int from) {
  for (int o = from; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Float64 block sums of (a, b) over the first nw warps (the warps that own nodes; the others
// hold zeros), valid in every lane of warp 0: for blocks whose sums are not for fixed point.
// Those threads park their values in shared memory; warp 0 adds them with a and b packed into
// the two half-warps, so each level of the dependence chain is one float64 warp instruction
// for both sums.
__device__ __noinline__ double2 rs_block_sum2(double a, double b, double* s_park, int nw) {
  if (threadIdx.x < 32 * nw) {
    s_park[threadIdx.x] = a;
    s_park[kRsThreads + threadIdx.x] = b;
  }
  __syncthreads();
  double2 t = make_double2(0.0, 0.0);
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x, h = lane & 15;
    const double* src = s_park + (lane < 16 ? 0 : kRsThreads);
    const int nv = 2 * nw;  // values per lane
    double v[kRsThreads / 16];
#pragma unroll
    for (int u = 0; u < kRsThreads / 16; ++u) v[u] = u < nv ? src[h + 16 * u] : 0.0;
#pragma unroll
    for (int w = 1; w < kRsThreads / 16; w *= 2)
#pragma unroll
      for (int u = 0; u + w < kRsThreads / 16; u += 2 * w)
        if (u + w < nv) v[u] += v[u + w];
    const double r = rs_xor_sum(v[0], 8);
    t = make_double2(__shfl_sync(0xffffffffu, r, 0), __shfl_sync(0xffffffffu, r, 16));
  }
  return t;
}

// ---- sums of r.r and w.r as integers ----
// A float64 warp instruction occupies the narrow FP64 pipe for 64 clocks and a level of a
// float64 tree takes at least that; a step of a small level is a chain of such levels.  The
// threads' partial sums are therefore brought to one power of two and added as integers: in a
// warp by three 32-bit reductions of 19-bit pieces, over the warps of a block, over the blocks
// (a warp's share of them, then the warps).  Every block adds the same integers, so the sums
// are the same in every block.  The power of two is that of the largest value added, anew at
// every level: a term is rounded to 2^-53 of the largest one or better, and to 2^-58 where the
// terms are of one size (a float64 sum rounds to 2^-53 of itself at every addition).

// A sum v 2^e; e = kRsRaw: v holds the bits of a float64 sum (infinities, NaN, extreme
// exponents, float64 solves); e = -kRsRaw: 0.  A block's part is two of them, r.r and w.r.
struct alignas(16) RsSum {
  long long v;
  int e, pad;
};
constexpr int kRsRaw = 1 << 20;
constexpr int kRsBits = 57;  // of a term: 32 of them fit 62 bits

// x as an integer of scale 2^(kRsBits - (E - 1022)), rounded; |x| < 2^(E - 1022).  0 for E < 64:
// below 2^-958, where the grid's largest |r|^2 is above 2^-846.
__device__ __forceinline__ long long rs_fixed(double x, int E) {
  if (E < 64) return 0;
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  // one bit below the unit, for rounding
  unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(x)) << (kRsBits - 53 + 1);
  const int d = min(E - e, 63);
  m = ((m >> d) + 1) >> 1;
  return hi < 0 ? -(long long)m : (long long)m;
}

// The warp's sum of v, |v| <= 2^57, in every lane.
__device__ __forceinline__ long long rs_warp_sum(long long v) {
  const int c0 = __reduce_add_sync(0xffffffffu, (int)(v & 0x7ffff));
  const int c1 = __reduce_add_sync(0xffffffffu, (int)((v >> 19) & 0x7ffff));
  const int c2 = __reduce_add_sync(0xffffffffu, (int)(v >> 38));
  return ((long long)c2 << 38) + ((long long)c1 << 19) + c0;
}

// v 2^-n, rounded.
__device__ __forceinline__ long long rs_round(long long v, int n) {
  n = min(n, 62);
  return (v + ((1LL << n) >> 1)) >> n;
}

// v 2^e as float64, v = 0 or the result a normal number (what the blocks' scales allow).
__device__ __forceinline__ double rs_double(long long v, int e) { return fx_scale((double)v, e); }

__device__ __forceinline__ RsSum rs_none() {
  RsSum t;
  t.v = 0;
  t.e = -kRsRaw;
  t.pad = 0;
  return t;
}

// Warp 0, after a block barrier: the sums of the warps' 2 x 8 sums (|v| <= 2^62), r.r in lanes 0
// .. 7 and w.r in lanes 8 .. 15: |v| <= 2^62.
__device__ __forceinline__ RsSum rs_over_warps(const RsSum (*s_warp)[kRsThreads / 32]) {
  static_assert(kRsThreads / 32 == 8, "eight warps");
  RsSum t = (&s_warp[0][0])[threadIdx.x & 15];
  const bool raw = t.e == kRsRaw;
  if (__any_sync(0xffffffffu, raw)) {
    double x = raw ? __longlong_as_double(t.v) : t.v ? rs_double(t.v, t.e) : 0.0;
#pragma unroll
    for (int o = 1; o < 8; o *= 2) x += __shfl_xor_sync(0xffffffffu, x, o);
    t.v = __double_as_longlong(x);
    t.e = kRsRaw;
    return t;
  }
  int m = t.e;
#pragma unroll
  for (int o = 1; o < 8; o *= 2) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  t.v = rs_round(t.v, m - t.e + 3);
#pragma unroll
  for (int o = 1; o < 8; o *= 2) t.v += __shfl_xor_sync(0xffffffffu, t.v, o);
  t.e = m + 3;
  return t;
}

// v 2^e of 56 bits (2^55 <= |v| <= 2^56, or none): two parts per lane are added.
__device__ __forceinline__ RsSum rs_norm(RsSum t) {
  if (t.e == kRsRaw) return t;
  if (t.v == 0) return rs_none();
  const int s = __clzll(t.v < 0 ? -t.v : t.v) - 1;
  t.v = rs_round(t.v << s, 7);
  t.e += 7 - s;
  return t;
}

// Reduction number `seq` (1, 2, ...): lanes 0 and 8 of warp 0 store this block's sums as part b
// of the set seq & 1 (two sets: a block can be one reduction ahead of another's reads, never
// two), thread 0 arrives on the counter with release semantics -- which also publishes every
// global store the block's threads made before the block barrier that precedes this
// call -- and waits (bounded) until all G blocks have arrived.  Returns, in every
// thread, false if the wait ran out or another block reported a time-out.
__device__ bool rs_arrive_wait(const RsSum& part, RsSum* parts, unsigned* counter, int G, unsigned seq,
                               int* err, int* s_ok) {
  if (threadIdx.x < 32) {
    if ((threadIdx.x & 23) == 0)
      __stcg(reinterpret_cast<int4*>(&parts[2 * ((size_t)(seq & 1) * G + blockIdx.x) + (threadIdx.x >> 3)]),
             reinterpret_cast<const int4&>(part));
    __syncwarp();
  }
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
    const unsigned target = seq * (unsigned)G;
    int ok = 1;
    unsigned long long spins = 0;
    while (ld_acquire_u32(counter) < target) {
      if (++spins > kRsSpinLimit || *(volatile int*)err) {
        ok = 0;
        break;
      }
      if (spins > 4096) __nanosleep(64);
    }
    if (!ok) atomicExch(err, 1);
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// The warp's sum of two terms per lane, |v| <= 2^56, identical in every lane: brought to the
// largest exponent and added as integers, or, where one is float64, all as float64 in a fixed
// order.
__device__ __forceinline__ RsSum rs_warp_terms(const RsSum& a, const RsSum& b) {
  RsSum t = rs_none();
  if (__any_sync(0xffffffffu, a.e == kRsRaw || b.e == kRsRaw)) {
    auto f = [](const RsSum& s) {
      return s.e == kRsRaw ? __longlong_as_double(s.v) : s.v ? rs_double(s.v, s.e) : 0.0;
    };
    t.v = __double_as_longlong(rs_xor_sum(f(a) + f(b), 16));
    t.e = kRsRaw;
    return t;
  }
  t.e = __reduce_max_sync(0xffffffffu, max(a.e, b.e));
  t.v = rs_warp_sum(rs_round(a.v, t.e - a.e) + rs_round(b.v, t.e - b.e));
  return t;
}

// After the wait, every warp: the sums of its share of the G parts of set seq & 1 into
// s_warp (then a block barrier).
__device__ __forceinline__ void rs_read_parts(const RsSum* parts, int G, unsigned seq,
                                              RsSum (*s_warp)[kRsThreads / 32]) {
  const RsSum* set = parts + 2 * (size_t)(seq & 1) * G;
  RsSum v[2][2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = threadIdx.x + u * kRsThreads;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      v[k][u] = rs_none();
      if (i < G) reinterpret_cast<int4&>(v[k][u]) = __ldcg(reinterpret_cast<const int4*>(set + 2 * i + k));
    }
  }
  const RsSum g = rs_warp_terms(v[0][0], v[0][1]), d = rs_warp_terms(v[1][0], v[1][1]);
  if ((threadIdx.x & 31) == 0) {
    s_warp[0][threadIdx.x >> 5] = g;
    s_warp[1][threadIdx.x >> 5] = d;
  }
}

// Warp 0, after that barrier: the sums, identical in every lane and every block.
__device__ __forceinline__ double2 rs_sums(const RsSum (*s_warp)[kRsThreads / 32]) {
  const RsSum t = rs_over_warps(s_warp);
  // both conversions in one warp instruction
  const double x = t.e == kRsRaw ? __longlong_as_double(t.v) : t.v ? rs_double(t.v, t.e) : 0.0;
  return make_double2(__shfl_sync(0xffffffffu, x, 0), __shfl_sync(0xffffffffu, x, 8));
}

// 19-point A-stencil at offset 0 of P with strides (1, ey, ez).  `shallow`: the seven
// weighted terms as a tree (two more float64 instructions, three fewer levels of
// dependence) -- for boxes of at most one node per thread, where a step waits on the
// chain rather than on the FP64 pipe's throughput.
__device__ __forceinline__ double rs_stencil(const double* P, int ey, int ez, const Coef& A,
                                             bool shallow) {
  const double SX = P[-1] + P[1], SY = P[-ey] + P[ey], SZ = P[-ez] + P[ez];
  const double EXY = (P[-1 - ey] + P[1 - ey]) + (P[-1 + ey] + P[1 + ey]);
  const double EXZ = (P[-1 - ez] + P[1 - ez]) + (P[-1 + ez] + P[1 + ez]);
  const double EYZ = (P[-ey - ez] + P[ey - ez]) + (P[-ey + ez] + P[ey + ez]);
  if (shallow) {
    const double t1 = fma(A.c0, P[0], A.fx * SX), t2 = fma(A.fy, SY, A.fz * SZ);
    const double t3 = fma(A.exy, EXY, A.exz * EXZ);
    return (t1 + t2) + fma(A.eyz, EYZ, t3);
  }
  return fma(A.c0, P[0], fma(A.fx, SX, fma(A.fy, SY, fma(A.fz, SZ, fma(A.exy, EXY, fma(A.exz, EXZ, A.eyz * EYZ))))));
}

// 2 LHS at offset 0 of the integers P with strides (1, ey, ez) (fixed_point.cuh).
__device__ __forceinline__ long long rs_stencil_fx(const long long* P, int ey, int ez, const FxWeights& W) {
  const long long SX = P[-1] + P[1], SY = P[-ey] + P[ey], SZ = P[-ez] + P[ez];
  const long long EXY = (P[-1 - ey] + P[1 - ey]) + (P[-1 + ey] + P[1 + ey]);
  const long long EXZ = (P[-1 - ez] + P[1 - ez]) + (P[-1 + ez] + P[1 + ez]);
  const long long EYZ = (P[-ey - ez] + P[ey - ez]) + (P[-ey + ez] + P[ey + ez]);
  const long long Q = ((SX + SY) + (SZ + (P[0] << 3))) << 1;
  return fx_weigh((EXY + EXZ - Q) + 10 * SX, (EXY + EYZ - Q) + 10 * SY, (EXZ + EYZ - Q) + 10 * SZ, W);
}

// Whether a node and its six neighbours, integers of the box's scale, all lie more than kFxRangeCG
// powers of two below it (|v| < 2^(kFxBits - 1 - kFxRangeCG), in either sign): by the high words,
// and by the low ones where those leave it open.  (With four neighbours white noise took a
// block to float64 every few steps.)
__device__ __forceinline__ bool rs_far_below(const long long* P, int ey, int ez) {
  constexpr int T = 1 << (kFxBits - 1 - kFxRangeCG - 32);
  auto hi = [&](int o) { return (int)(P[o] >> 32); };
  const int top = max(hi(0), max(max(max(hi(-1), hi(1)), max(hi(-ey), hi(ey))), max(hi(-ez), hi(ez))));
  const int low = min(hi(0), min(min(min(hi(-1), hi(1)), min(hi(-ey), hi(ey))), min(hi(-ez), hi(ez))));
  if (top >= T || low < -T) return false;
  if (low > -T) return true;
  constexpr long long t = -((long long)T << 32);
  return !(P[0] == t || P[-1] == t || P[1] == t || P[-ey] == t || P[ey] == t || P[-ez] == t || P[ez] == t);
}

// ONE: boxes of at most one node per thread, whose vectors stay in the threads' registers;
// else they are in shared memory.
template <bool ONE>
__global__ void __launch_bounds__(kRsThreads, 2)
    k_cg_resident(const ResidentDesc D, CGState* st, RsSum* parts, unsigned* counter, int* err) {
  extern __shared__ __align__(16) double s_vec[];
  __shared__ double s_park[2 * kRsThreads];
  __shared__ uint4 s_mag[kRsThreads / 128];
  // r.r and w.r of each warp: of its nodes, then of its share of the blocks
  __shared__ RsSum s_warp[2][kRsThreads / 32];
  __shared__ int s_ok;
  __shared__ double s_alpha, s_beta;
  __shared__ int s_stop;
  CGState* S = st + D.slot;
  if (S->done) return;  // identical in every block: the state is written after the last wait
  const Grid3 g = D.g;
  const int G = gridDim.x;
  const int BX = D.bx, BY = D.by, BZ = D.bz;
  const int EX = BX + 2, EY = BY + 2, EZ = BZ + 2;
  const int B = BX * BY * BZ, ext = EX * EY * EZ;
  const int nw_own = min(kRsThreads, B + 31) / 32;  // warps that own nodes
  const int b = blockIdx.x;
  const int ibx = b % D.nbx, iby = (b / D.nbx) % D.nby, ibz = b / (D.nbx * D.nby);
  // global node of box-local (0, 0, 0); the halo starts one node before
  const int i0 = 1 + ibx * BX, j0 = 1 + iby * BY, k0 = 1 + ibz * BZ;
  // r of the box and its halo as integers of the block's scale (or float64 bits):
  // (lx+1) + EX (ly+1) + EX EY (lz+1); then r, x, p, s, w of the box
  long long* RI = reinterpret_cast<long long*>(s_vec);
  double* R = s_vec + ext;
  double* X = R + B;
  double* P = X + B;
  double* Sv = P + B;
  double* W = Sv + B;
  const Coef A = D.A;
  const FxWeights FW = D.W;
  // own node q of the box: its index in RI and in the level's node array; valid = the
  // node exists (boxes at the far faces of the grid may be partial)
  struct Own {
    int e;
    bool valid;
    long long o;
  };
  const int sx = 31 - __clz(BX), sxy = sx + 31 - __clz(BY);  // box extents are powers of two
  auto own_node = [&](int q) -> Own {
    const int lx = q & (BX - 1), ly = (q >> sx) & (BY - 1), lz = q >> sxy;
    const int gi = i0 + lx, gj = j0 + ly, gk = k0 + lz;
    Own w;
    w.e = (lx + 1) + EX * ((ly + 1) + EY * (lz + 1));
    w.o = gi + gj * g.sy + (long long)gk * g.sz;
    w.valid = q < B && gi < g.nx && gj < g.ny && gk < g.nz;
    return w;
  };
  // ONE: this thread's node, computed once (the index arithmetic divides by the box extents)
  // instead of in every step, and its vectors
  const Own mine = own_node(threadIdx.x);
  double xr = 0.0, xx = 0.0, xp = 0.0, xs = 0.0, xw = 0.0;
  // every own node of this thread: f(node, r, x, p, s, w)
  auto each = [&](auto f) {
    if (ONE) {
      if (mine.valid) f(mine, xr, xx, xp, xs, xw);
    } else {
      // (unrolled, the stencil's loop: 11.7 us a step on 64^3, 11.3 as it is)
#pragma unroll 1
      for (int q = threadIdx.x; q < B; q += kRsThreads) {
        const Own n = own_node(q);
        if (n.valid) f(n, R[q], X[q], P[q], Sv[q], W[q]);
      }
    }
  };
  // shell position h (0 .. ext - B - 1): the 2 z-faces, then the 2 y-faces, then the 2
  // x-faces of the extended box
  const int zf = EX * EY, yf = EX * BZ, xf = BY * BZ;
  const int nshell = 2 * (zf + yf + xf);
  auto shell_node = [&](int h, int& e, int& gi, int& gj, int& gk) {
    int ex, ey, ez;
    if (h < 2 * zf) {
      ez = h < zf ? 0 : EZ - 1;
      const int r = h % zf;
      ex = r % EX;
      ey = r / EX;
    } else if (h < 2 * (zf + yf)) {
      const int h2 = h - 2 * zf;
      ey = h2 < yf ? 0 : EY - 1;
      const int r = h2 % yf;
      ex = r % EX;
      ez = 1 + r / EX;
    } else {
      const int h3 = h - 2 * (zf + yf);
      ex = h3 < xf ? 0 : EX - 1;
      const int r = h3 % xf;
      ey = 1 + r % BY;
      ez = 1 + r / BY;
    }
    e = ex + EX * (ey + EY * ez);
    gi = i0 - 1 + ex;
    gj = j0 - 1 + ey;
    gk = k0 - 1 + ez;
  };
  auto interior = [&](int gi, int gj, int gk) {
    return gi > 0 && gi < g.nx && gj > 0 && gj < g.ny && gk > 0 && gk < g.nz;
  };
  // this thread's shell nodes (index in RI, offset in the level's arrays or -1 outside the
  // interior), computed once: after each wait the loads issue at once
  // (the slots past `slots` hold none)
  const int slots = min(kRsHB, (nshell + kRsThreads - 1) / kRsThreads);
  int he[kRsHB], ho[kRsHB];
#pragma unroll
  for (int u = 0; u < kRsHB; ++u) {
    const int h = threadIdx.x + u * kRsThreads;
    he[u] = -1;
    ho[u] = -1;
    if (h < nshell) {
      int gi, gj, gk;
      shell_node(h, he[u], gi, gj, gk);
      if (interior(gi, gj, gk)) ho[u] = gi + gj * g.sy + gk * g.sz;
    }
  }
  // The halo's new r of shells of more than kRsHB per thread: value(o) of the interior nodes, as
  // float64 bits into RI; returns the largest magnitude word.
  auto shell_rest = [&](auto value) -> unsigned {
    unsigned m = 0;
    for (int h = threadIdx.x + kRsHB * kRsThreads; h < nshell; h += kRsThreads) {
      int e, gi, gj, gk;
      shell_node(h, e, gi, gj, gk);
      const double v = interior(gi, gj, gk) ? value(gi + gj * g.sy + (long long)gk * g.sz) : 0.0;
      RI[e] = __double_as_longlong(v);
      m = max(m, fx_mag(v));
    }
    return m;
  };
  // put(v) of the new r to the box: own (each thread its r) and halo hn.
  auto put_box = [&](const double (&hn)[kRsHB], auto put) {
    each([&](const Own& n, double& r, double&, double&, double&, double&) { RI[n.e] = put(r); });
#pragma unroll
    for (int u = 0; u < kRsHB; ++u) {
      if (u >= slots) break;
      if (he[u] >= 0) RI[he[u]] = put(hn[u]);
    }
  };
  // The box of integers from the new r: own, halo hn (and, of larger shells, the float64 bits
  // already in RI); mag: this thread's largest magnitude word.  Returns the scale E, or -1 for
  // a box of float64 bits.  Two barriers.
  auto fill = [&](unsigned mag, const double (&hn)[kRsHB]) -> int {
    mag = __reduce_max_sync(0xffffffffu, mag);
    if ((threadIdx.x & 31) == 0) reinterpret_cast<unsigned*>(s_mag)[threadIdx.x >> 5] = mag;
    __syncthreads();
    const uint4 m0 = s_mag[0], m1 = s_mag[1];
    mag = max(max(max(m0.x, m0.y), max(m0.z, m0.w)), max(max(m1.x, m1.y), max(m1.z, m1.w)));
    // r.r and w.r stay in the normal range too
    int E = (int)(mag >> 20);
    const int q = fx_sum_exp(FW.k, E);
    if (E < 600 || E > 1400 || q < -400 || q > 300 || D.float64) E = -1;
    auto put = [&](double v) { return E < 0 ? __double_as_longlong(v) : fx_from_double<kFxBits>(v, E); };
    put_box(hn, put);
    for (int h = threadIdx.x + kRsHB * kRsThreads; h < nshell; h += kRsThreads) {
      int e, gi, gj, gk;
      shell_node(h, e, gi, gj, gk);
      RI[e] = put(__longlong_as_double(RI[e]));
    }
    __syncthreads();
    return E;
  };
  // w = A r of the box (published to Wn), and the block's sums of r.r and w.r in lanes 0 and 8
  // of warp 0.  A box with a node that lies, with its neighbours, far below the box's scale is
  // taken again in float64, as one without a scale (value: shell_rest's).
  auto apply = [&](int E, const double (&hn)[kRsHB], auto value, double* Wn) -> RsSum {
    RsSum part = rs_none();
    double acc_g = 0.0, acc_d = 0.0;
    if (E >= 0) {
      const int qL = fx_sum_exp(FW.k, E) - 1;
      bool far = false;
      each([&](const Own& n, double& r, double&, double&, double&, double& w) {
        far |= rs_far_below(RI + n.e, EX, EX * EY);
        w = fx_scale_neg((double)rs_stencil_fx(RI + n.e, EX, EX * EY, FW), qL);
        acc_g = fma(r, r, acc_g);
        acc_d = fma(w, r, acc_d);
        __stcg(Wn + n.o, w);
      });
      // the warp's sums, at the exponents of its largest terms
      auto expo = [](double x) { return (__double2hiint(x) >> 20) & 0x7ff; };
      const int xg = __reduce_max_sync(0xffffffffu, expo(acc_g)), xd = __reduce_max_sync(0xffffffffu, expo(acc_d));
      const long long sg = rs_warp_sum(rs_fixed(acc_g, xg)), sd = rs_warp_sum(rs_fixed(acc_d, xd));
      if ((threadIdx.x & 31) == 0) {
        part.v = sg;
        part.e = sg ? xg - 1022 - kRsBits : -kRsRaw;
        s_warp[0][threadIdx.x >> 5] = part;
        part.v = sd;
        part.e = sd ? xd - 1022 - kRsBits : -kRsRaw;
        s_warp[1][threadIdx.x >> 5] = part;
      }
      if (!__syncthreads_or(far)) {
        if (threadIdx.x < 32) part = rs_norm(rs_over_warps(s_warp));
        return part;
      }
      put_box(hn, [](double v) { return __double_as_longlong(v); });
      shell_rest(value);
      __syncthreads();
      acc_g = acc_d = 0.0;
    }
    each([&](const Own& n, double& r, double&, double&, double&, double& w) {
      w = rs_stencil(reinterpret_cast<const double*>(RI) + n.e, EX, EX * EY, A, ONE);
      acc_g = fma(r, r, acc_g);
      acc_d = fma(w, r, acc_d);
      __stcg(Wn + n.o, w);
    });
    const double2 t = rs_block_sum2(acc_g, acc_d, s_park, nw_own);
    part.v = __double_as_longlong((threadIdx.x & 31) < 8 ? t.x : t.y);
    part.e = kRsRaw;
    return part;
  };
  // the published r, w, s of up to kRsHB halo nodes per thread, loaded right after each
  // reduction's wait, so that the load latency overlaps the reading of the partials and
  // the scalar arithmetic (zero on the boundary)
  double hr[kRsHB], hw[kRsHB], hs[kRsHB];
  auto load_halo = [&](int par) {
    const double* Rg = par ? D.r1 : D.r;
    const double* Wg = par ? D.w1 : D.w0;
    const double* Sg = par ? D.s1 : D.s0;
#pragma unroll
    for (int u = 0; u < kRsHB; ++u) {
      hr[u] = hw[u] = hs[u] = 0.0;
      if (ho[u] >= 0) {
        hr[u] = __ldcg(Rg + ho[u]);
        hw[u] = __ldcg(Wg + ho[u]);
        hs[u] = __ldcg(Sg + ho[u]);
      }
    }
  };
  // ---- start: r_0 on the box and its halo, x; p = s = 0; w_0 = A r_0; publish w_0, s = 0
  for (int e = threadIdx.x; e < ext; e += kRsThreads) RI[e] = 0;
  __syncthreads();
  unsigned mag = 0;
  each([&](const Own& n, double& r, double& x, double& p, double& s, double& w) {
    r = D.r[n.o];
    x = D.x[n.o];
    p = s = w = 0.0;
    D.s0[n.o] = 0.0;
    mag = max(mag, fx_mag(r));
  });
#pragma unroll
  for (int u = 0; u < kRsHB; ++u) {
    hr[u] = ho[u] >= 0 ? D.r[ho[u]] : 0.0;
    mag = max(mag, fx_mag(hr[u]));
  }
  auto start = [&](long long o) { return D.r[o]; };
  mag = max(mag, shell_rest(start));
  RsSum part = apply(fill(mag, hr), hr, start, D.w0);
  // CG scalars: warp 0 keeps identical copies in all its lanes (and in every block)
  double gam = S->rr, alpha = 0.0, beta = 0.0, delta = 0.0;
  const double tol2 = S->tol2;
  int iter = S->iter;
  const int max_iter = S->max_iter, fixed = S->fixed;
  int status = EXCMG_OK;
  const int lane = threadIdx.x & 31;
  unsigned seq = 1;
  {
    const bool ok = rs_arrive_wait(part, parts, counter, G, seq, err, &s_ok);
    if (ok) {
      load_halo(0);
      rs_read_parts(parts, G, seq, s_warp);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      int stop = 0;
      if (!ok) {
        status = EXCMG_ERR_TIMEOUT;
        stop = 1;
      } else {
        delta = rs_sums(s_warp).y;
        if (delta == 0.0 && gam == 0.0) {
          stop = 1;  // exact solution (fixed-count mode)
        } else if (!(delta > 0.0) || !isfinite(delta)) {
          status = EXCMG_ERR_NONFINITE;
          stop = 1;
        } else {
          alpha = gam / delta;
        }
      }
      if (lane == 0) {
        s_stop = stop;
        s_alpha = alpha;
        s_beta = 0.0;
      }
    }
    ++seq;
    __syncthreads();
  }
  int par = 0;  // step i reads the published r_i, w_i, s_{i-1} of parity par
  while (!s_stop) {
    const double a = s_alpha, bt = s_beta;
    const double* Rg = par ? D.r1 : D.r;
    const double* Wg = par ? D.w1 : D.w0;
    const double* Sg = par ? D.s1 : D.s0;
    double* Rn = par ? D.r : D.r1;
    double* Wn = par ? D.w0 : D.w1;
    double* Sn = par ? D.s0 : D.s1;
    // 1. own nodes: p, s, x, r; publish r and s
    mag = 0;
    each([&](const Own& n, double& r, double& x, double& p, double& s, double& w) {
      const double pv = fma(bt, p, r), sv = fma(bt, s, w);
      p = pv;
      s = sv;
      x = fma(a, pv, x);
      const double rn = fma(-a, sv, r);
      r = rn;
      mag = max(mag, fx_mag(rn));
      __stcg(Rn + n.o, rn);
      __stcg(Sn + n.o, sv);
    });
    // 2. the halo's new r, with the owner's fused operations; shells larger than kRsHB
    // per thread finish with plain loads
    double hn[kRsHB];
#pragma unroll
    for (int u = 0; u < kRsHB; ++u) {
      if (u >= slots) break;  // (a float64 instruction takes its 64 clocks with every lane predicated off too)
      hn[u] = fma(-a, fma(bt, hs[u], hw[u]), hr[u]);  // 0 where there is no node: hr, hw, hs are
      mag = max(mag, fx_mag(hn[u]));
    }
    // (the arrays read here stay as they are until every block has arrived below)
    auto value = [&](long long o) { return fma(-a, fma(bt, __ldcg(Sg + o), __ldcg(Wg + o)), __ldcg(Rg + o)); };
    mag = max(mag, shell_rest(value));
    // 3. w = A r, gamma, delta; publish w
    part = apply(fill(mag, hn), hn, value, Wn);
    // 4. the grid reduction (it also orders every block's publications before the next
    // step's halo loads); the next halo's loads; scalars
    const bool ok = rs_arrive_wait(part, parts, counter, G, seq, err, &s_ok);
    par ^= 1;
    if (ok) {
      rs_read_parts(parts, G, seq, s_warp);
      load_halo(par);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      int stop = 0;
      if (!ok) {
        status = EXCMG_ERR_TIMEOUT;
        stop = 1;
      } else {
        const double2 red = rs_sums(s_warp);
        const double gn = red.x, dn = red.y;
        iter += 1;
        if (b == 0 && lane == 0 && D.hist && iter < D.hist_len) D.hist[iter] = gn;
        if (!isfinite(gn) || !isfinite(dn)) {
          status = EXCMG_ERR_NONFINITE;
          stop = 1;
        } else if (gn <= tol2 || gn == 0.0) {
          stop = 1;  // converged (or exact solution in fixed-count mode)
        } else if (iter >= max_iter) {
          if (!fixed) status = EXCMG_ERR_NOT_CONVERGED;
          stop = 1;
        } else {
          // alpha' = gn / (dn - beta' gn / alpha) = gn k / (dn k - gn^2), k = gam alpha;
          // beta' = gn / gam: both divides in one instruction (lanes 0 and 1)
          const double k = gam * alpha;
          const double den = fma(dn, k, -gn * gn);
          if (!(den > 0.0)) {
            status = EXCMG_ERR_NONFINITE;
            stop = 1;
          } else {
            const double q = (lane == 0 ? gn * k : gn) / (lane == 0 ? den : gam);
            alpha = __shfl_sync(0xffffffffu, q, 0);
            beta = __shfl_sync(0xffffffffu, q, 1);
          }
        }
        gam = gn;
        delta = dn;
      }
      if (lane == 0) {
        s_stop = stop;
        s_alpha = alpha;
        s_beta = beta;
      }
    }
    ++seq;
    __syncthreads();
  }
  // x and the last r of the box
  each([&](const Own& n, double& r, double& x, double&, double&, double&) {
    D.x[n.o] = x;
    D.r[n.o] = r;
  });
  if (b == 0 && threadIdx.x == 0) {
    S->rr = gam;
    S->pq = delta;
    S->alpha = alpha;
    S->beta = beta;
    S->iter = iter;
    S->first = 0;
    S->status = status;
    S->done = 1;
  }
}

int g_rs_blocks_per_sm = 0;  // at the largest shared memory a box may take
int g_rs_sms = 0;
size_t g_rs_max_smem = 0;

}  // namespace

size_t resident_smem(int bx, int by, int bz) {
  const size_t ext = (size_t)(bx + 2) * (by + 2) * (bz + 2), nodes = (size_t)bx * by * bz;
  return sizeof(double) * (ext + (nodes > kRsThreads ? 5 * nodes : 0));
}

#ifndef EXCMG_RESIDENT_MAX_SMEM
#define EXCMG_RESIDENT_MAX_SMEM (107 * 1024)  // two blocks of an SM, with 5 KB each of their own
#endif

bool resident_box(const Grid3& g, ResidentDesc& D, size_t& smem) {
  if (g_rs_sms == 0) {
    int dev = 0, coop = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&g_rs_sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    g_rs_max_smem = std::min<size_t>(EXCMG_RESIDENT_MAX_SMEM, (size_t)std::max(0, optin - 2048));
    if (!coop || g_rs_sms <= 0 ||
        cudaFuncSetAttribute(k_cg_resident<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)g_rs_max_smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_rs_blocks_per_sm, k_cg_resident<false>, kRsThreads,
                                                      g_rs_max_smem) != cudaSuccess) {
      cudaGetLastError();
      g_rs_blocks_per_sm = 0;
    }
    if (g_rs_sms <= 0) g_rs_sms = 1;
  }
  if (g_rs_blocks_per_sm <= 0) return false;
  const int ni = g.nx - 1, nj = g.ny - 1, nk = g.nz - 1;
  if (ni < 1 || nj < 1 || nk < 1) return false;
  // (a block reads at most two sums per thread)
  const long long max_blocks = std::min<long long>((long long)g_rs_sms * g_rs_blocks_per_sm, 2 * kRsThreads);
  // per-step model in SM clocks: the busiest SM's float64 work (~12.5 clocks per node,
  // 2 DFMA per clock, plus ~400 per block for its reduction), the halo loads of a box
  // (3 per shell node), and the grid reduction's share per block (arrival, partials).  The
  // constants are those of the sums in float64 and were not fitted anew to the integer ones.
  double best = 1e300;
  bool found = false;
  const int bxs[] = {32, 16, 8};
  const int bys[] = {1, 2, 4, 8, 16, 32};
  const int bzs[] = {1, 2, 4, 8, 16, 32};
  for (int bx : bxs)
    for (int by : bys)
      for (int bz : bzs) {
        const long long nb = (long long)((ni + bx - 1) / bx) * ((nj + by - 1) / by) * ((nk + bz - 1) / bz);
        if (nb > max_blocks) continue;
        const size_t sm = resident_smem(bx, by, bz);
        if (sm > g_rs_max_smem) continue;
        const double B = (double)bx * by * bz;
        const double shell = (double)(bx + 2) * (by + 2) * (bz + 2) - B;
        const double per_sm = (double)((nb + g_rs_sms - 1) / g_rs_sms);
        const double cost = per_sm * (B * 12.5 + 400.0) + shell * 6.0 + (double)nb * 12.0;
        if (cost < best) {
          best = cost;
          found = true;
          D.bx = bx;
          D.by = by;
          D.bz = bz;
          D.nbx = (ni + bx - 1) / bx;
          D.nby = (nj + by - 1) / by;
          D.nbz = (nk + bz - 1) / bz;
          smem = sm;
        }
      }
  return found;
}

cudaError_t launch_cg_resident(const ResidentDesc& D, size_t smem, CGState* st, void* parts,
                               unsigned* counter, int* err, cudaStream_t s) {
  const int grid = D.nbx * D.nby * D.nbz;
  ResidentDesc d = D;
  void* args[] = {(void*)&d, (void*)&st, (void*)&parts, (void*)&counter, (void*)&err};
  const bool one = D.bx * D.by * D.bz <= kRsThreads;
  return cudaLaunchCooperativeKernel(one ? (const void*)k_cg_resident<true> : (const void*)k_cg_resident<false>, dim3(grid), dim3(kRsThreads), args,
                                     smem, s);
}

}  // namespace excmg
