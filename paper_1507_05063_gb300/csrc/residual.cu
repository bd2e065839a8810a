// The residual of the 19-point compact scheme (Section 2, eqs. compact and FD):
// r = LHS(u) - RHS(f) = b - A u_I, with r.r, b.b and the start of a level's CG state.
//
// The sums run in block fixed point (fixed_point.cuh, fixed_slab.cuh): a float64 form needs
// about 23 float64 instructions per node, 11.5 clocks of an SM at 2 lanes per clock, ten
// times the 24 bytes a node moves.  Here five remain (the two conversions of the sums, the
// difference, r.r and RHS.RHS).  Measured, one call on 320 x 255 x 257 cells: 1.11 ms in
// float64, 0.44 ms here (the kernel 380 us; float64 pipe 58% busy, issue slots 50%), 1.16 to 1.18
// where every slab is taken again in float64 (u = exp(-100 x), exp(-200 r^2)).  Error of r against
// 128-bit arithmetic, root mean square, float64 / here: exp(x + y + z) on 64^3 cells 3.1e-11 /
// 4.9e-15, on 48 x 100 x 37 4.7e-11 / 3.9e-13, r^{5/3} on 64^3 5.3e-12 / 5.6e-15, white noise 9.9e-12 /
// 6.8e-12, exp(-100 x) 2.3e-13 / 2.4e-13.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "block_reduce.cuh"
#include "excmg_internal.cuh"
#include "fixed_slab.cuh"

namespace excmg {

namespace {

struct FinRes {
  const ResDesc* descs;
  CGState* st;
  __device__ void operator()(int p, const double* s) const {
    const ResDesc& d = descs[p];
    CGState& S = st[d.slot];
    const double rr = s[0];
    // s[1] = ||b||^2 (lift included), s[2] = ||RHS(f)||^2: the two readings of ||f_h||
    const double bb = !d.want_b ? S.bb : (d.forcing && s[2] > 0.0) ? s[2] : s[1];
    S.rr = rr;
    S.rr0 = rr;
    S.bb = bb;
    S.alpha = 0.0;
    S.beta = 0.0;
    S.pq = 0.0;
    S.iter = 0;
    S.first = 1;
    S.max_iter = d.max_iter;
    S.fixed = d.fixed;
    S.status = EXCMG_OK;
    S.tol2 = d.fixed ? -1.0 : fmax(d.tol_b2 * bb, d.tol_r2 * rr);
    if (d.hist && d.hist_len > 0) d.hist[0] = rr;
    S.done = d.fixed ? (d.max_iter <= 0) : (rr <= S.tol2 || d.max_iter <= 0);
    // no step allowed and the start does not pass the test: the level is unconverged
    if (!d.fixed && d.max_iter <= 0 && !(rr <= S.tol2)) S.status = EXCMG_ERR_NOT_CONVERGED;
    if (!isfinite(rr) || !isfinite(bb)) {
      S.status = EXCMG_ERR_NONFINITE;
      S.done = 1;
    }
  }
};

// The Dirichlet lift of an interior node next to the boundary: the part of its 19-point
// A-sum over boundary nodes.
__device__ __noinline__ double node_lift(const double* __restrict__ u, const Grid3& g, const Coef& A, int i, int j,
                                         int k) {
  const double* c = u + i + j * g.sy + k * g.sz;
  const bool bx[3] = {i == 1, false, i == g.nx - 1}, by[3] = {j == 1, false, j == g.ny - 1},
             bz[3] = {k == 1, false, k == g.nz - 1};
  // u at (dx, dy, dz) from the node if that is a boundary node, else 0
  auto B = [&](int dx, int dy, int dz) {
    return bx[dx + 1] || by[dy + 1] || bz[dz + 1] ? __ldg(c + dx + dy * g.sy + dz * g.sz) : 0.0;
  };
  const double SX = B(-1, 0, 0) + B(1, 0, 0), SY = B(0, -1, 0) + B(0, 1, 0), SZ = B(0, 0, -1) + B(0, 0, 1);
  const double EXY = (B(-1, -1, 0) + B(1, -1, 0)) + (B(-1, 1, 0) + B(1, 1, 0));
  const double EXZ = (B(-1, 0, -1) + B(1, 0, -1)) + (B(-1, 0, 1) + B(1, 0, 1));
  const double EYZ = (B(0, -1, -1) + B(0, 1, -1)) + (B(0, -1, 1) + B(0, 1, 1));
  return fma(A.fx, SX, fma(A.fy, SY, A.fz * SZ)) + fma(A.exy, EXY, fma(A.exz, EXZ, A.eyz * EYZ));
}

// RHS(f) of eq. (compact) at interior node (i, j, k) in float64: 3 f_c + half the 6 face
// values of f, or the value an earlier pass kept, or -b when b is given directly.  o is
// the node's offset.
__device__ __forceinline__ double res_rhs(const ResDesc& d, int i, int j, int k, long long o) {
  if (d.rhs_in != nullptr) return d.rhs_in[o];
  if (d.src != nullptr) return -d.src[o];
  const View& F = d.f;
  return fma(3.0, F.at(i, j, k), 0.5 * ((F.at(i - 1, j, k) + F.at(i + 1, j, k)) +
                                        (F.at(i, j - 1, k) + F.at(i, j + 1, k)) +
                                        (F.at(i, j, k - 1) + F.at(i, j, k + 1))));
}

// The residual's block sums of one problem (r.r, ||b||^2 with the lift, ||RHS(f)||^2)
// added to its three partials in shared memory.  Called at problem switches only; kept
// out of line so that it adds no registers to the plane loop.
__device__ __noinline__ void residual_flush(double acc_r, double acc_b, double acc_f, double* part) {
  const double v[3] = {acc_r, acc_f + acc_b, acc_f};
  const double s = block_sums(v);
  if ((threadIdx.x & 31) == 0 && threadIdx.x < 96) part[threadIdx.x >> 5] += s;
}

// lift (lift + 2 RHS) of the interior nodes x0 .. x1 - 1 (y, z likewise) of a slab that are
// next to a boundary face, in one pass over the faces' nodes (a node next to several faces
// belongs to the first of z, y, x).
__device__ __noinline__ double slab_lift(const ResDesc& d, int x0, int y0, int z0, int x1, int y1, int z1) {
  const Grid3& g = d.g;
  const int wx = x1 - x0, wy = y1 - y0, wz = z1 - z0;
  // the planes next to a face that the slab holds: 0, 1 or 2 per direction (at 1 and n - 1)
  const bool zl = z0 == 1, zh = z1 == g.nz && (g.nz > 2 || !zl), yl = y0 == 1, yh = y1 == g.ny && (g.ny > 2 || !yl);
  const bool xl = x0 == 1, xh = x1 == g.nx && (g.nx > 2 || !xl);
  const int nzf = (zl + zh) * wx * wy, nyf = (yl + yh) * wx * wz, nxf = (xl + xh) * wy * wz;
  double acc = 0.0;
  for (int t = threadIdx.x; t < nzf + nyf + nxf; t += kThreads) {
    int i, j, k;
    if (t < nzf) {
      const int s = t / (wx * wy), r = t - s * (wx * wy);
      k = zl && s == 0 ? 1 : g.nz - 1;
      i = x0 + r % wx;
      j = y0 + r / wx;
    } else if (t < nzf + nyf) {
      const int t2 = t - nzf, s = t2 / (wx * wz), r = t2 - s * (wx * wz);
      j = yl && s == 0 ? 1 : g.ny - 1;
      i = x0 + r % wx;
      k = z0 + r / wx;
      if (k == 1 || k == g.nz - 1) continue;
    } else {
      const int t3 = t - nzf - nyf, s = t3 / (wy * wz), r = t3 - s * (wy * wz);
      i = xl && s == 0 ? 1 : g.nx - 1;
      j = y0 + r % wy;
      k = z0 + r / wy;
      if (k == 1 || k == g.nz - 1 || j == 1 || j == g.ny - 1) continue;
    }
    const double lift = node_lift(d.u, g, d.A, i, j, k);
    const double rhs = res_rhs(d, i, j, k, i + j * g.sy + k * g.sz);
    acc = fma(lift, fma(2.0, rhs, lift), acc);
  }
  return acc;
}

__device__ __forceinline__ void put_r(double* p, double v) { *p = v; }
__device__ __forceinline__ void put_r(float* p, double v) { *p = fx_to_float(v); }

struct ResSmem {
  FxSmem u;  // u's box; the magnitude words of u and f
  long long f[kFxG * kPlane];
};

// What one slab adds to the block's sums.
struct ResSums {
  double r = 0.0, f = 0.0;  // r.r, RHS.RHS
};

// One slab: r on its interior nodes, RHS(f) kept where asked.  TF: RHS(f) is formed here,
// else read (d.rhs_in, or -d.src).  F64: the sums in float64.  Returns false, in every
// thread, when a group is not for fixed point (the caller then takes the slab again with
// F64).  All threads of the block must call.
template <typename TR, bool TF, bool F64>
__device__ __noinline__ bool residual_slab(const ResDesc& d, const FxSlab c, ResSmem& S, ResSums& sums) {
  const int nx = d.g.nx, ny = d.g.ny;
  const long long sy = d.g.sy, sz = d.g.sz;
  const FxCols C(c);
  // own nodes, and columns to load: nodes 0 .. n per direction
  const bool own = C.i < nx && C.j < ny, lown = C.i <= nx && C.j <= ny;
  bool rim[kRimT];
#pragma unroll
  for (int m = 0; m < kRimT; ++m) rim[m] = C.rim_box[m] >= 0 && C.rim_x[m] <= nx && C.rim_y[m] <= ny;
  // the group's addresses in u and f: own node of its first plane, rim nodes
  const double *pu = d.u + (C.i + C.j * sy + (c.z0 - 1) * sz), *pf = nullptr;
  const double *ru[kRimT], *rf[kRimT];
#pragma unroll
  for (int m = 0; m < kRimT; ++m) ru[m] = d.u + (C.rim_x[m] + C.rim_y[m] * sy + (c.z0 - 1 + C.rim_z[m]) * sz);
  const long long fz = d.f.sz;
  if (TF) {
    const View& F = d.f;
    pf = F.p + (C.i * F.sx + C.j * F.sy + (c.z0 - 1) * fz);
#pragma unroll
    for (int m = 0; m < kRimT; ++m) rf[m] = F.p + (C.rim_x[m] * F.sx + C.rim_y[m] * F.sy + (c.z0 - 1 + C.rim_z[m]) * fz);
  }
  const long long osy = sizeof(TR) == 4 ? d.osy : sy, osz = sizeof(TR) == 4 ? d.osz : sz;
  TR* __restrict__ rout = reinterpret_cast<TR*>(d.r) + (C.i + C.j * osy + c.z0 * osz);
  const long long o0 = C.i + C.j * sy + c.z0 * sz;
  double* __restrict__ kept = TF && d.rhs_out ? d.rhs_out + o0 : nullptr;
  const double* __restrict__ given = TF ? nullptr : (d.rhs_in ? d.rhs_in : d.src) + o0;
  double next = !TF && own ? *given : 0.0;  // RHS given: of the next plane, loaded one ahead
  const int flip = !TF && !d.rhs_in ? (int)0x80000000 : 0;  // RHS = -src
  const bool want_b = d.want_b != 0;
  const FxWeights W = d.W;
  FxMarch M;
  F64March D;
  // f of the last plane, and 6 f with its faces but the one above
  using FT = typename std::conditional<F64, double, long long>::type;
  FT f1 = 0, s1 = 0;
  FxRange U, V;  // of u and f
  double acc_r = 0.0, acc_f = 0.0;
  auto ld = [](const double* a) { return __ldg(a); };
  for (int k0 = c.z0 - 1; k0 <= c.z1; k0 += kFxG) {
    double v[kLoads];
    bool held = true;
    if (TF) {
      load_group(v, pf, lown, rf, rim, C, fz, 0, c.z1 - k0, ld);
      pf += kFxG * fz;
#pragma unroll
      for (int m = 0; m < kRimT; ++m) rf[m] += kFxG * fz;
      if (!F64) warp_mag(v, own, c.z1 - 1 - k0, S.u.mag[1]);
      __syncthreads();  // the boxes of the group before are read
      if (F64) {
        store_box(reinterpret_cast<double*>(S.f), v, C, [](double x) { return x; });
      } else {
        const int was = V.scale;
        if (!V.next(S.u.mag[1])) return false;
        held = V.near(S.u.mag[1], kFxRange);
        const int sf = V.scale;
        if (sf != was) {
          f1 = (FT)fx_shift((long long)f1, was - sf);
          s1 = (FT)fx_shift((long long)s1, was - sf);
        }
        store_box(S.f, v, C, [&](double x) { return fx_from_double<kFxBitsF>(x, sf); });
      }
    }
    load_group(v, pu, lown, ru, rim, C, sz, 0, c.z1 - k0, ld);
    pu += kFxG * sz;
#pragma unroll
    for (int m = 0; m < kRimT; ++m) ru[m] += kFxG * sz;
    if (!F64) warp_mag(v, own, c.z1 - 1 - k0, S.u.mag[0]);
    if (!F64 || !TF) __syncthreads();
    if (F64) {
      store_box(reinterpret_cast<double*>(S.u.box), v, C, [](double x) { return x; });
    } else {
      const int was = U.scale;
      if (!U.next(S.u.mag[0])) return false;
      held = held & U.near(S.u.mag[0], kFxRange);
      const int su = U.scale;
      if (su != was) M.rescale(was - su);
      store_box(S.u.box, v, C, [&](double x) { return fx_from_double<kFxBits>(x, su); });
    }
    const int qL = fx_sum_exp(W.k, U.scale) - 1, qF = V.scale - 1022 - kFxBitsF - 1;  // LHS = L 2^qL, RHS = F 2^qF
    if (!F64 && (!held || qL < -1000 || qL > 900)) return false;
    const double scale = fx_pow2(qL);
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < kFxG; ++s) {
      const bool in = k0 + s > c.z0 && k0 + s <= c.z1;  // this plane completes the sums of the one before
      const bool out = in && own;
      double now = 0.0;
      if (!TF && out) {
        now = __hiloint2double(__double2hiint(next) ^ flip, __double2loint(next));
        given += sz;
        if (k0 + s < c.z1) next = *given;
      }
      FT g0 = 0, gs = 0;  // f of this plane, and its in-plane faces
      if (TF) {
        const FT* b = reinterpret_cast<const FT*>(S.f) + s * kPlane + fx_corner();
        g0 = b[kBoxX + 1];
        gs = (b[kBoxX] + b[kBoxX + 2]) + (b[1] + b[2 * kBoxX + 1]);
      }
      auto put = [&](double lhs_or_Au) {  // F64: A u, else L
        double rhs = now;
        if (TF) {
          if constexpr (F64)
            rhs = 0.5 * (s1 + g0);
          else
            rhs = fx_scale((double)(s1 + g0), qF);
        }
        const double rv = F64 ? -rhs - lhs_or_Au : fma(lhs_or_Au, scale, -rhs);
        if (TF && kept) {
          *kept = rhs;
          kept += sz;
        }
        if (want_b) acc_f = fma(rhs, rhs, acc_f);
        acc_r = fma(rv, rv, acc_r);
        put_r(rout, rv);
        rout += osz;
      };
      if (F64)
        D.plane(reinterpret_cast<const double*>(S.u.box) + s * kPlane + fx_corner(), d.A, [&](double, double Au) {
          if (out) put(Au);
        });
      else
        M.plane(S.u.box + s * kPlane + fx_corner(), W, [&](long long, auto lhs2) {
          if (out) put((double)lhs2());
        });
      if (TF) {
        s1 = gs + (6 * g0 + f1);
        f1 = g0;
      }
    }
  }
  sums.r += acc_r;
  sums.f += acc_f;
  return true;
}

template <typename TR>
__device__ __forceinline__ void residual_slab_any(const ResDesc& d, const FxSlab& c, ResSmem& S, ResSums& sums) {
  if (d.rhs_in || d.src) {
    if (d.float64 || !residual_slab<TR, false, false>(d, c, S, sums)) residual_slab<TR, false, true>(d, c, S, sums);
  } else {
    if (d.float64 || !residual_slab<TR, true, false>(d, c, S, sums)) residual_slab<TR, true, true>(d, c, S, sums);
  }
}

// r = 0 on the grid's boundary nodes, by block bl of G: a row per warp (no divisions: they
// took a third of a small grid's prologue).
template <typename TR>
__device__ __noinline__ void zero_r_faces(const ResDesc& d, int bl, int G) {
  const Grid3& g = d.g;
  const long long osy = sizeof(TR) == 4 ? d.osy : g.sy, osz = sizeof(TR) == 4 ? d.osz : g.sz;
  TR* r = reinterpret_cast<TR*>(d.r);
  const int lane = threadIdx.x & 31, warp = bl * (kThreads / 32) + (threadIdx.x >> 5), nw = G * (kThreads / 32);
  for (int j = warp; j <= g.ny; j += nw)
    for (int i = lane; i <= g.nx; i += 32) r[i + j * osy] = r[i + j * osy + g.nz * osz] = (TR)0.0;
  for (int k = warp; k <= g.nz; k += nw) {
    for (int i = lane; i <= g.nx; i += 32) r[i + k * osz] = r[i + k * osz + g.ny * osy] = (TR)0.0;
    for (int j = lane; j <= g.ny; j += 32) r[j * osy + k * osz] = r[j * osy + k * osz + g.nx] = (TR)0.0;
  }
}

// TR: the type r is stored in (float: MIXED inner solves).
template <typename TR>
__global__ void __launch_bounds__(kThreads, kFxBlocks)
    k_residual(int nprob, const ResDesc* __restrict__ descs, long long total_tiles, CGState* st,
               double* partials, unsigned* counters) {
  __shared__ ResSmem S;
  __shared__ int s_active[kMaxProb];
  __shared__ double s_part[3 * kMaxProb];
  for (int p = threadIdx.x; p < nprob; p += blockDim.x) {
    s_active[p] = 1;
    s_part[3 * p] = 0.0;
    s_part[3 * p + 1] = 0.0;
    s_part[3 * p + 2] = 0.0;
  }
  __syncthreads();
  for (int p = 0; p < nprob; ++p) zero_r_faces<TR>(descs[p], blockIdx.x, gridDim.x);
  int cur = -1, p = 0;
  // sums.f sums RHS^2 over every interior node: the forcing reading of ||f_h||^2.  b =
  // -RHS - lift, and the lift is nonzero only next to the boundary, so ||b||^2 = sums.f +
  // acc_b with acc_b summing b^2 - RHS^2 = lift (lift + 2 RHS) over those nodes (the lift
  // reading).
  ResSums sums;
  double acc_b = 0.0;
  for (long long t = blockIdx.x; t < total_tiles; t += gridDim.x) {
    p = find_problem(descs, nprob, t, p);
    if (p != cur) {
      if (cur >= 0) residual_flush(sums.r, acc_b, sums.f, s_part + 3 * cur);
      sums = ResSums();
      acc_b = 0.0;
      cur = p;
    }
    const ResDesc& d = descs[p];
    const FxSlab c = fx_slab(d.g, d.t, t - d.tile_begin);
    residual_slab_any<TR>(d, c, S, sums);
    if (d.want_b) {
      const int x1 = min(c.x0 + kFxX, d.g.nx), y1 = min(c.y0 + kFxY, d.g.ny);
      if (c.x0 == 1 || c.y0 == 1 || c.z0 == 1 || x1 == d.g.nx || y1 == d.g.ny || c.z1 == d.g.nz)
        acc_b += slab_lift(d, c.x0, c.y0, c.z0, x1, y1, c.z1);
    }
  }
  if (cur >= 0) residual_flush(sums.r, acc_b, sums.f, s_part + 3 * cur);
  __syncthreads();
  publish_and_finish<3>(nprob, s_active, s_part, partials, counters, FinRes{descs, st});
}

int device_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(1, sms);
  }
  return sms;
}

}  // namespace

Tiling make_fx_tiling(const Grid3& g, int tz) {
  Tiling t;
  t.tz = tz;
  t.ntx = (g.nx - 1 + kFxX - 1) / kFxX;
  t.nty = (g.ny - 1 + kFxY - 1) / kFxY;
  t.ntz = (g.nz - 1 + tz - 1) / tz;
  return t;
}

// The depth that minimises the busiest SM's time, over the even cuts of the deepest grid.
// A full round of slabs takes kFxBlocks units of an SM's time per plane, a last round of k
// slabs per SM k units (at least three: fewer wait on their own latency); a slab's planes
// count with its two halo planes, in groups of six, and about two planes' time for its start.
int choose_fx_tz(const Grid3* grids, int n) {
  const long long sms = device_sms();
  int deepest = 1;
  for (int k = 0; k < n; ++k) deepest = std::max(deepest, grids[k].nz - 1);
  int best = 2;
  double best_cost = 1e300;
  for (int cuts = 1; cuts <= 256; ++cuts) {
    const int tz = (deepest + cuts - 1) / cuts;
    if (tz < 2 && cuts > 1) break;
    long long slabs = 0;
    for (int k = 0; k < n; ++k) slabs += make_fx_tiling(grids[k], tz).count();
    const long long full = slabs / (kFxBlocks * sms), rest = slabs - full * kFxBlocks * sms;
    const long long last = (rest + sms - 1) / sms;
    const double units = (double)(full * kFxBlocks) + (rest > 0 ? std::max<double>((double)last, 3.0) : 0.0);
    const double cost = units * ((tz + 2 + kFxG - 1) / kFxG * kFxG + 2);
    if (cost < best_cost) {
      best_cost = cost;
      best = tz;
    }
  }
  return best;
}

// The depth that minimises the longest team's step, over the even cuts of the deepest grid: a
// team has a block per slab if all slabs get one, else its share of the blocks (cg_loop's
// rule), and its slabs per block take their planes as in choose_fx_tz.
int choose_team_tz(const Grid3* grids, int n, int blocks) {
  int deepest = 1;
  for (int k = 0; k < n; ++k) deepest = std::max(deepest, grids[k].nz - 1);
  int best = 2;
  double best_cost = 1e300;
  for (int cuts = 1; cuts <= 256; ++cuts) {
    const int tz = (deepest + cuts - 1) / cuts;
    if (tz < 2 && cuts > 1) break;
    long long slabs = 0, rounds = 1;
    for (int k = 0; k < n; ++k) slabs += make_fx_tiling(grids[k], tz).count();
    for (int k = 0; k < n && slabs > blocks; ++k) {
      const long long tp = make_fx_tiling(grids[k], tz).count(), share = std::max(1LL, tp * blocks / slabs);
      rounds = std::max(rounds, (tp + share - 1) / share);
    }
    const double cost = (double)rounds * ((tz + 2 + kFxG - 1) / kFxG * kFxG + 2);
    if (cost < best_cost) {
      best_cost = cost;
      best = tz;
    }
  }
  return best;
}

FxWeights make_fx_weights(const Grid3& g) {
  const double w[3] = {1.0 / (g.hx * g.hx), 1.0 / (g.hy * g.hy), 1.0 / (g.hz * g.hz)};
  int ex = 0;
  frexp(std::max(w[0], std::max(w[1], w[2])), &ex);
  FxWeights W;
  if (!(w[0] + w[1] + w[2] < 1e300 && w[0] + w[1] + w[2] > 1e-300)) {
    W = FxWeights{{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, 1 << 20};  // no tile's range holds: the float64 form
    return W;
  }
  W.k = 60 - ex;  // the largest weight becomes 2^59 .. 2^60
  for (int d = 0; d < 3; ++d) {
    const long long v = llrint(ldexp(w[d], W.k));
    W.l[d] = (int)((v + (1LL << 30)) & 0x7fffffffLL) - (1 << 30);
    W.l2[d] = 2 * W.l[d];
    W.h[d] = (int)((v - W.l[d]) >> 31);
  }
  return W;
}

cudaError_t launch_residual(bool out_float, int nprob, const ResDesc* descs, long long total_tiles, CGState* st,
                            double* partials, unsigned* counters, cudaStream_t s) {
  // all co-resident blocks, at most one per slab; three partials per block have
  // room for 2 x kMaxGrid
  const int most = std::min(kFxBlocks * device_sms(), 2 * kMaxGrid / 3);
  const int grid = (int)std::max(1LL, std::min<long long>(total_tiles, most));
  if (out_float)
    k_residual<float><<<grid, kThreads, 0, s>>>(nprob, descs, total_tiles, st, partials, counters);
  else
    k_residual<double><<<grid, kThreads, 0, s>>>(nprob, descs, total_tiles, st, partials, counters);
  return cudaGetLastError();
}

}  // namespace excmg
