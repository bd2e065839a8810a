// Slabs of the fixed-point stencil kernels (residual.cu, the float64 CG of cg_kernels.cu).
//
// A slab is 32 x 8 columns of interior nodes, its first (1 + 32 a, 1 + 8 b), over tz planes
// from 1 + tz c: a direction of 2^k cells (2^k - 1 interior nodes) has no ragged slab but
// the last.  A block of 256 threads, one per column, marches it along z in groups of six
// planes: a thread loads its 6 nodes of a group and at most 2 of the group's x- and y-halo,
// the group is brought to one scale, stored as 64-bit integers in shared memory (16 KB) and
// summed; the partial sums of the last planes stay in registers from group to group, so
// nothing is loaded or converted twice along z but the slab's two halo planes.  Three blocks
// of an SM (80 registers) cover each other's loads and barriers.  Measured slower: two rows
// per thread (fewer shared-memory reads, but spills or fewer warps), and the next group's
// loads held in registers (two blocks per SM).
//
// The scale of a group is the largest exponent of its planes and the previous group's (whose
// last two planes its sums still hold): the sums carried over are shifted when it changes.
// Where a neighbourhood of the group is far smaller than the scale, its values would be held in
// fewer bits than their own size asks for: such a slab takes the float64 form (FxRange).
#pragma once

#include "excmg_internal.cuh"
#include "fixed_point.cuh"

namespace excmg {
namespace {

constexpr int kFxX = kTX, kFxY = kThreads / 32;
// Planes per group: 84 rim nodes a plane go to 256 threads, so groups of 3 and 6 planes fill
// the loads' rounds and others do not, and a deeper group has fewer barriers.  Residual at
// 320 x 255 x 257 with 3 / 4 / 5 / 6 / 7 / 8 planes: 475 / 455 / 422 / 421 / 452 / 424 us; CG at
// 385 x 201 x 121, 40 steps: 4.39 / 4.39 / 4.24 / 4.15 / 4.30 / 4.88 ms (without FxRange's check).
constexpr int kFxG = 6;
constexpr int kBoxX = kFxX + 2, kBoxY = kFxY + 2;
constexpr int kPlane = kBoxX * kBoxY;
constexpr int kOwn = kFxG;                                         // own nodes per thread and group
constexpr int kRim = kPlane - kFxX * kFxY;                         // halo nodes of a plane
constexpr int kRimT = (kRim * kFxG + kThreads - 1) / kThreads;     // ... of a group, per thread
constexpr int kLoads = kOwn + kRimT;
static_assert(kFxX == 32 && kFxY == kFxSlabY, "one warp per x-run of a slab row");

struct FxMags {
  uint4 top[kThreads / 128];    // a word per warp: warp_mag
  unsigned low[kThreads / 32];
};
struct FxSmem {
  FxMags mag[2];  // of two arrays
  long long box[kFxG * kPlane];
};

struct FxSlab {
  int x0, y0, z0, z1;  // first own node; one past the last own plane
};

__device__ __forceinline__ FxSlab fx_slab(const Grid3& g, const Tiling& tl, long long lt) {
  FxSlab c;
  // (a grid that fits the memory has fewer than 2^32 slabs of 512 nodes and more)
  const unsigned r = (unsigned)lt / (unsigned)tl.ntx, z = r / (unsigned)tl.nty;
  c.x0 = 1 + (int)((unsigned)lt - r * (unsigned)tl.ntx) * kFxX;
  c.y0 = 1 + (int)(r - z * (unsigned)tl.nty) * kFxY;
  c.z0 = 1 + (int)z * tl.tz;
  c.z1 = min(c.z0 + tl.tz, g.nz);
  return c;
}

// This thread's nodes of a slab's plane groups: its own column (i, j), and rim nodes at
// (x, y) of plane z of a group, at rim_box of the box (-1: none).
struct FxCols {
  int i, j, rim_x[kRimT], rim_y[kRimT], rim_z[kRimT], rim_box[kRimT];
  __device__ __forceinline__ explicit FxCols(const FxSlab& c) {
    i = c.x0 + (threadIdx.x & 31);
    j = c.y0 + (threadIdx.x >> 5);
#pragma unroll
    for (int m = 0; m < kRimT; ++m) {
      const int h = threadIdx.x + m * kThreads, p = h / kRim, r = h - p * kRim;
      int x, y;
      if (r < 2 * kBoxX) {
        y = r < kBoxX ? 0 : kBoxY - 1;
        x = r < kBoxX ? r : r - kBoxX;
      } else {
        const int r2 = r - 2 * kBoxX;
        x = r2 < kFxY ? 0 : kBoxX - 1;
        y = 1 + (r2 < kFxY ? r2 : r2 - kFxY);
      }
      rim_x[m] = c.x0 - 1 + x;
      rim_y[m] = c.y0 - 1 + y;
      rim_z[m] = p;
      rim_box[m] = p < kFxG ? p * kPlane + y * kBoxX + x : -1;
    }
  }
};

// This thread's share of a group from a node array: own, rim: its nodes' addresses in the
// group's first plane (the rim's in its own plane); planes lo .. hi of the group hold data,
// the others zeros.
template <typename Ld>
__device__ __forceinline__ void load_group(double (&v)[kLoads], const double* own, bool has_own,
                                           const double* const (&rim)[kRimT], const bool (&has_rim)[kRimT],
                                           const FxCols& C, long long sz, int lo, int hi, const Ld& ld) {
  if (lo <= 0 && hi >= kFxG - 1) {
#pragma unroll
    for (int n = 0; n < kOwn; ++n) v[n] = has_own ? ld(own + n * sz) : 0.0;
#pragma unroll
    for (int m = 0; m < kRimT; ++m) v[kOwn + m] = has_rim[m] ? ld(rim[m]) : 0.0;
  } else {
#pragma unroll
    for (int n = 0; n < kOwn; ++n) v[n] = has_own && n >= lo && n <= hi ? ld(own + n * sz) : 0.0;
#pragma unroll
    for (int m = 0; m < kRimT; ++m)
      v[kOwn + m] = has_rim[m] && C.rim_z[m] >= lo && C.rim_z[m] <= hi ? ld(rim[m]) : 0.0;
  }
}

// This thread's own node of a box plane, and the corner of its 3 x 3 neighbourhood.
__device__ __forceinline__ int fx_corner() { return (threadIdx.x >> 5) * kBoxX + (threadIdx.x & 31); }

// put(v) of every loaded value to its place in the box.
template <typename T, typename Put>
__device__ __forceinline__ void store_box(T* box, const double (&v)[kLoads], const FxCols& C, const Put& put) {
  T* b = box + fx_corner() + kBoxX + 1;
#pragma unroll
  for (int n = 0; n < kOwn; ++n) b[n * kPlane] = put(v[n]);
#pragma unroll
  for (int m = 0; m < kRimT; ++m)
    if (C.rim_box[m] >= 0) box[C.rim_box[m]] = put(v[kOwn + m]);
}

// This warp's magnitude words of a group (a block barrier, then FxRange): the largest of its
// values, and the smallest of its own nodes' neighbourhoods (~0: no own nodes).  A
// neighbourhood is four planes (0 .. 3 or 2 .. 5 of the group) of a column and the columns
// beside it; `own`: the thread has a column of interior nodes; last: the slab's last own plane
// in the group.
__device__ __forceinline__ void warp_mag(const double (&v)[kLoads], bool own, int last, FxMags& S) {
  static_assert(kFxG == 6, "two overlapping windows of four planes");
  unsigned m = 0;
#pragma unroll
  for (int k = kOwn; k < kLoads; ++k) m = max(m, fx_mag(v[k]));
  const unsigned mid = max(fx_mag(v[2]), fx_mag(v[3]));
  unsigned a = max(mid, max(fx_mag(v[0]), fx_mag(v[1]))), b = max(mid, max(fx_mag(v[4]), fx_mag(v[5])));
  m = __reduce_max_sync(0xffffffffu, max(m, max(a, b)));
  a = max(a, max(__shfl_up_sync(0xffffffffu, a, 1), __shfl_down_sync(0xffffffffu, a, 1)));
  b = max(b, max(__shfl_up_sync(0xffffffffu, b, 1), __shfl_down_sync(0xffffffffu, b, 1)));
  const unsigned l = __reduce_min_sync(0xffffffffu, min(own && last >= 0 ? a : ~0u, own && last >= 2 ? b : ~0u));
  if (m == 0) {  // all zero, or denormal below 2^-1042: not for fixed point
    unsigned lo = 0;
#pragma unroll
    for (int k = 0; k < kLoads; ++k) lo |= (unsigned)__double2loint(v[k]);
    m = __any_sync(0xffffffffu, lo != 0);
  }
  if ((threadIdx.x & 31) == 0) {
    reinterpret_cast<unsigned*>(S.top)[threadIdx.x >> 5] = m;
    S.low[threadIdx.x >> 5] = l;
  }
}

// The scales of a slab's groups: a group's is the largest exponent of its planes and the
// previous group's.
struct FxRange {
  int E = 0, low = 4095, scale = kFxMinExp;
  // The scale of the next group; false, in every thread, where its exponents are outside
  // [kFxMinExp, kFxMaxExp].
  __device__ __forceinline__ bool next(const FxMags& S) {
    static_assert(kThreads == 256, "eight words of two 16-byte reads");
    const uint4 a = S.top[0], b = S.top[1];
    const unsigned m = max(max(max(a.x, a.y), max(a.z, a.w)), max(max(b.x, b.y), max(b.z, b.w)));
    const int was = E;
    E = (int)(m >> 20);
    scale = max(max(E, was), kFxMinExp);
    return m == 0 || (E >= kFxMinExp && E <= kFxMaxExp);
  }
  // (After next.)  Whether the group's and the previous group's values are held near their own
  // size: false, in every thread, if all values of a neighbourhood (of three columns, three rows and four
  // planes) lie more than `range` powers of two below the scale, in a group that is not all
  // zero.
  __device__ __forceinline__ bool near(const FxMags& S, int range) {
    const unsigned l = S.low[threadIdx.x & 7], h = l == ~0u ? 0 : l;
    // a row's neighbourhoods, or those of a row beside it
    const unsigned h3 = max(h, max(__shfl_up_sync(0xffffffffu, h, 1, 8), __shfl_down_sync(0xffffffffu, h, 1, 8)));
    const int was = low;
    low = (int)(__reduce_min_sync(0xffffffffu, l == ~0u || E == 0 ? ~0u : h3) >> 20);
    return scale - min(low, was) <= range;
  }
};

// x 2^d: to the left exactly (the caller knows it fits), to the right to nearest, ties to even.
__device__ __forceinline__ long long fx_shift(long long x, int d) {
  if (d >= 0) return x << min(d, 63);
  const int s = min(-d, 62);
  const long long y = x + ((1LL << s) >> 1);
  return (y >> s) & ~(long long)((y & ((1LL << s) - 1)) == 0);
}

// The march of a thread's column.  With S_x, S_y, E a plane's in-plane neighbour and edge
// sums of a node of value c, the three sums of fixed_point.cuh are, per plane k,
//   X_k = (E + 10 S_x - 2 w)_k + (S_x - 2 c)_{k-1} + (S_x - 2 c)_{k+1},   w = 8 c + S_x + S_y,
//   Y_k likewise with S_y,   Z_k = w_{k-1} - 2 w_k + w_{k+1}:
// what plane k + 1 adds is what plane k added to plane k - 1's sums, so a plane is read once
// and three partial sums, the three terms and (for p.q) c stay in registers.
struct FxMarch {
  long long c1 = 0, px = 0, py = 0, pz = 0, tx = 0, ty = 0, tw = 0;
  __device__ __forceinline__ void rescale(int d) {
    c1 = fx_shift(c1, d);
    px = fx_shift(px, d);
    py = fx_shift(py, d);
    pz = fx_shift(pz, d);
    tx = fx_shift(tx, d);
    ty = fx_shift(ty, d);
    tw = fx_shift(tw, d);
  }
  // Takes the next plane (s: this thread's corner of it); emit(c, L) gets the value c and
  // 2 LHS (a call: nodes that need none cost none) of the plane before.
  template <typename Emit>
  __device__ __forceinline__ void plane(const long long* s, const FxWeights& W, const Emit& emit) {
    const long long sm = s[0] + s[2], sx = s[kBoxX] + s[kBoxX + 2], sp = s[2 * kBoxX] + s[2 * kBoxX + 2];
    const long long c = s[kBoxX + 1], sy = s[1] + s[2 * kBoxX + 1];
    const long long w = (sx + sy) + (c << 3), ax = sx - (c << 1), ay = sy - (c << 1);
    emit(c1, [&]() { return fx_weigh(px + ax, py + ay, pz + w, W); });
    const long long w2 = w << 1, b = (sm + sp) - w2;
    px = (b + tx) + 10 * sx;
    py = (b + ty) + 10 * sy;
    pz = tw - w2;
    tx = ax;
    ty = ay;
    tw = w;
    c1 = c;
  }
};

// The same march in float64 (the box holds doubles): per plane the in-plane part C = c0 P +
// fx S_x + fy S_y + exy E_xy and the out-of-plane part T = fz P + exz S_x + eyz S_y of the
// 19-point sum of A, (A u)_k = C_k + T_{k-1} + T_{k+1}: 14 operations per node.
struct F64March {
  double p1 = 0.0, c1 = 0.0, t1 = 0.0, t2 = 0.0;
  // emit(p, Ap) of the plane before
  template <typename Emit>
  __device__ __forceinline__ void plane(const double* s, const Coef& A, const Emit& emit) {
    const double sm = s[0] + s[2], sx = s[kBoxX] + s[kBoxX + 2], sp = s[2 * kBoxX] + s[2 * kBoxX + 2];
    const double p = s[kBoxX + 1], sy = s[1] + s[2 * kBoxX + 1];
    const double Ck = fma(A.c0, p, fma(A.fx, sx, fma(A.fy, sy, A.exy * (sm + sp))));
    const double Tk = fma(A.fz, p, fma(A.exz, sx, A.eyz * sy));
    emit(p1, (c1 + t2) + Tk);
    t2 = t1;
    t1 = Tk;
    c1 = Ck;
    p1 = p;
  }
};

}  // namespace
}  // namespace excmg
