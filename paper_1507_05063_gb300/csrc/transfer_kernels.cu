// Level-to-level transfers of Algorithm 1 (Section 3.3):
//   EXP_finite(u_2h, u_4h) -> w_h   (the initial guess; eqs. jiedian, zhongdian, inter)
//   EXP_true(u_h, u_2h)    -> u~_h  (the optional last step; eqs. t1, chenlin)
// and the adjoint's transposed right-hand-side / lift operators.
//
// EXP_finite works on bricks of 32 x 8 x 8 fine cells (four interpolation cells along x,
// each cell = 2x2x2 elements of grid 4h = 8 fine cells per direction).  Per brick:
//  1. w at every node of grid 2h: u_2h + (1/16) * (mean of d = u_2h - u_4h over the
//     grid-4h corners of the edge / face / element it is the centre of; d itself at a
//     grid-4h node).  This is eq. (jiedian) at corners ((17u1 - u0)/16 = u1 + d/16),
//     eq. (zhongdian) at edge midpoints (u1 + (d_a + d_b)/32), and the arithmetic means
//     of eq. (zhongdian) over the two face diagonals / four space diagonals.  The corner
//     sums are formed separably (x, then y, then z: one add per odd coordinate) and the
//     power-of-two factor 1/(16 * 2^(number of odd coordinates)) is applied in one FMA;
//  2. tri-quartic interpolation (eq. inter) as three one-dimensional quartic passes
//     (x, then y, then z) with the Lagrange weights at the half-integer points of a cell:
//     the tensor product l_i(xi) l_j(eta) l_k(zeta) applied by sum factorisation, ~6 FMA
//     per node instead of the 125 of the 604x125 matrix form.
// Every pass splits its outputs by parity (copies at even positions, arithmetic at odd
// ones) so that the float64 work of a warp runs with all lanes active: on GB300 a warp
// instruction on the narrow FP64 pipe costs the same whether 16 or 32 lanes need it.
//
// The same brick code, instantiated with fewer interpolation points, gives the two
// comparison prolongations of the library's prolong option: the extrapolated grid-2h
// values interpolated tri-quadratically over cells of 2x2x2 grid-2h elements (the
// interpolation of the earlier EXCMG for linear elements, which the first remark of
// Section 3.3 contrasts with the tri-quartic one), and plain trilinear interpolation of
// u_2h with no extrapolation (the cascadic multigrid prolongation of Section 3).
#include <math.h>

#include <algorithm>

#include "excmg_internal.cuh"
#include "fixed_point.cuh"

namespace excmg {

namespace {

// 128 * l_m(t) for the five nodes t = 0..4 of a cell and t = 1/2, 3/2, 5/2, 7/2
// (Lagrange basis of Section 3.3; exact in binary floating point after / 128).
__constant__ double c_wq[4][5] = {
    {35.0 / 128, 140.0 / 128, -70.0 / 128, 28.0 / 128, -5.0 / 128},
    {-5.0 / 128, 60.0 / 128, 90.0 / 128, -20.0 / 128, 3.0 / 128},
    {3.0 / 128, -20.0 / 128, 90.0 / 128, 60.0 / 128, -5.0 / 128},
    {-5.0 / 128, 28.0 / 128, -70.0 / 128, 140.0 / 128, 35.0 / 128},
};

// 8 * l_m(t) of the quadratic basis on the nodes 0, 1, 2 at t = 1/2, 3/2, and the linear
// interpolation at the midpoint of two nodes (both exact in binary floating point).
__constant__ double c_wquad[2][3] = {{3.0 / 8, 6.0 / 8, -1.0 / 8}, {-1.0 / 8, 6.0 / 8, 3.0 / 8}};
__constant__ double c_wlin[1][2] = {{0.5, 0.5}};

constexpr int BX1 = 17, BY1 = 5, BZ1 = 5;  // grid-2h nodes of a brick
constexpr int BX0 = 9, BY0 = 3, BZ0 = 3;   // grid-4h nodes of a brick
constexpr int BXF = 33, BYF = 9, BZF = 9;  // fine nodes of a brick

struct BrickSmem {
  double wq[4][5];            // c_wq, indexed per lane
  double u1[BZ1][BY1][BX1];   // grid-2h values
  double tx[BZ0][BY0][BX1];   // corner sums of d along x (grid-4h rows, grid-2h columns)
  double ty[BZ0][BY1][BX1];   // ... then along y
  double w[BZ1][BY1][BX1];    // extrapolated values at the grid-2h nodes
  double x[BZ1][BY1][BXF];    // after the quartic pass along x
  double y[BZ1][BYF][BXF];    // after the quartic pass along y
};

// One brick (local index lb) of the prolongation for descriptor d.  P interpolation
// points per direction over cells of P - 1 grid-2h elements: 5 is EXP_finite (eq. inter);
// 3 the tri-quadratic comparison; 2 the trilinear one, which also skips the
// extrapolation (w = u_2h at the grid-2h nodes).  The brick (16 x 4 x 4 grid-2h
// elements) holds whole cells for each P.
template <int P>
__device__ void exp_finite_brick(const ProlongDesc& d, long long lb, BrickSmem& S) {
  constexpr int C = P - 1;  // grid-2h elements per cell and direction
  const Grid3 g = d.g;
  const int bx = (int)(lb % d.nbx);
  const int by = (int)((lb / d.nbx) % d.nby);
  const int bz = (int)(lb / ((long long)d.nbx * d.nby));
  const int n1x = g.nx / 2, n1y = g.ny / 2, n1z = g.nz / 2;
  const int n0x = g.nx / 4, n0y = g.ny / 4, n0z = g.nz / 4;
  const long long s1y = n1x + 1, s1z = (long long)(n1x + 1) * (n1y + 1);
  const long long s0y = n0x + 1, s0z = (long long)(n0x + 1) * (n0y + 1);
  // d = u_2h - u_4h at grid-4h node (I, J, K) of the level (0 outside the grid)
  auto dval = [&](int I, int J, int K) -> double {
    if (I > n0x || J > n0y || K > n0z) return 0.0;
    return d.u2h[2 * I + 2 * J * s1y + 2 * K * s1z] - d.u4h[I + J * s0y + K * s0z];
  };
  __syncthreads();  // shared buffers of the previous brick are free
  // 1a. stage grid-2h values; corner sums of d along x (even columns: d, odd: d_a + d_b)
  if (P == 2) {  // no extrapolation: w = u_2h
    for (int idx = threadIdx.x; idx < BZ1 * BY1 * BX1; idx += kThreads) {
      const int ix = idx % BX1, jy = (idx / BX1) % BY1, kz = idx / (BX1 * BY1);
      const int I = 16 * bx + ix, J = 4 * by + jy, K = 4 * bz + kz;
      S.w[kz][jy][ix] = (I <= n1x && J <= n1y && K <= n1z) ? d.u2h[I + J * s1y + K * s1z] : 0.0;
    }
  } else {
  for (int idx = threadIdx.x; idx < BZ1 * BY1 * BX1; idx += kThreads) {
    const int ix = idx % BX1, jy = (idx / BX1) % BY1, kz = idx / (BX1 * BY1);
    const int I = 16 * bx + ix, J = 4 * by + jy, K = 4 * bz + kz;
    S.u1[kz][jy][ix] = (I <= n1x && J <= n1y && K <= n1z) ? d.u2h[I + J * s1y + K * s1z] : 0.0;
  }
  for (int idx = threadIdx.x; idx < BZ0 * BY0 * BX0; idx += kThreads) {
    const int i0 = idx % BX0, j0 = (idx / BX0) % BY0, k0 = idx / (BX0 * BY0);
    S.tx[k0][j0][2 * i0] = dval(8 * bx + i0, 2 * by + j0, 2 * bz + k0);
  }
  for (int idx = threadIdx.x; idx < BZ0 * BY0 * (BX0 - 1); idx += kThreads) {
    const int i0 = idx % (BX0 - 1), j0 = (idx / (BX0 - 1)) % BY0, k0 = idx / ((BX0 - 1) * BY0);
    const int I = 8 * bx + i0, J = 2 * by + j0, K = 2 * bz + k0;
    S.tx[k0][j0][2 * i0 + 1] = dval(I, J, K) + dval(I + 1, J, K);
  }
  __syncthreads();
  // 1b. along y
  for (int idx = threadIdx.x; idx < BZ0 * BY0 * BX1; idx += kThreads) {
    const int ix = idx % BX1, j0 = (idx / BX1) % BY0, k0 = idx / (BX1 * BY0);
    S.ty[k0][2 * j0][ix] = S.tx[k0][j0][ix];
  }
  for (int idx = threadIdx.x; idx < BZ0 * (BY0 - 1) * BX1; idx += kThreads) {
    const int ix = idx % BX1, j0 = (idx / BX1) % (BY0 - 1), k0 = idx / (BX1 * (BY0 - 1));
    S.ty[k0][2 * j0 + 1][ix] = S.tx[k0][j0][ix] + S.tx[k0][j0 + 1][ix];
  }
  __syncthreads();
  // 1c. along z, and w = u_2h + sum / (16 * 2^(odd coordinates)) (a power of two: exact)
  for (int idx = threadIdx.x; idx < BZ0 * BY1 * BX1; idx += kThreads) {
    const int ix = idx % BX1, jy = (idx / BX1) % BY1, k0 = idx / (BX1 * BY1);
    const double scale = 0.0625 / (double)(1 << ((ix & 1) + (jy & 1)));
    S.w[2 * k0][jy][ix] = fma(S.ty[k0][jy][ix], scale, S.u1[2 * k0][jy][ix]);
  }
  for (int idx = threadIdx.x; idx < (BZ0 - 1) * BY1 * BX1; idx += kThreads) {
    const int ix = idx % BX1, jy = (idx / BX1) % BY1, k0 = idx / (BX1 * BY1);
    const double scale = 0.03125 / (double)(1 << ((ix & 1) + (jy & 1)));
    S.w[2 * k0 + 1][jy][ix] = fma(S.ty[k0][jy][ix] + S.ty[k0 + 1][jy][ix], scale, S.u1[2 * k0 + 1][jy][ix]);
  }
  }  // P != 2
  __syncthreads();
  // 2a. interpolation along x: even fine columns are grid-2h columns
  for (int idx = threadIdx.x; idx < BZ1 * BY1 * BX1; idx += kThreads) {
    const int ix = idx % BX1, jy = (idx / BX1) % BY1, kz = idx / (BX1 * BY1);
    S.x[kz][jy][2 * ix] = S.w[kz][jy][ix];
  }
  for (int idx = threadIdx.x; idx < BZ1 * BY1 * (BX1 - 1); idx += kThreads) {
    const int I = idx % (BX1 - 1), jy = (idx / (BX1 - 1)) % BY1, kz = idx / ((BX1 - 1) * BY1);
    const int t = I % C, base = I - t;
    double v = 0.0;
#pragma unroll
    for (int m = 0; m < P; ++m) v = fma(S.wq[t][m], S.w[kz][jy][base + m], v);
    S.x[kz][jy][2 * I + 1] = v;
  }
  __syncthreads();
  // 2b. along y (odd fine row 2q + 1 lies in the cell starting at grid-2h row q - q % C)
  for (int idx = threadIdx.x; idx < BZ1 * BY1 * BXF; idx += kThreads) {
    const int lx = idx % BXF, jy = (idx / BXF) % BY1, kz = idx / (BXF * BY1);
    S.y[kz][2 * jy][lx] = S.x[kz][jy][lx];
  }
  for (int idx = threadIdx.x; idx < BZ1 * (BY1 - 1) * BXF; idx += kThreads) {
    const int lx = idx % BXF, q = (idx / BXF) % (BY1 - 1), kz = idx / (BXF * (BY1 - 1));
    const int t = q % C, base = q - t;
    double v = 0.0;
#pragma unroll
    for (int m = 0; m < P; ++m) v = fma(S.wq[t][m], S.x[kz][base + m][lx], v);
    S.y[kz][2 * q + 1][lx] = v;
  }
  __syncthreads();
  // 2c. along z, boundary data, store.  Main part: the 32 x 8 x 8 nodes whose
  // brick-local coordinates are all below the brick's far faces -- one fine plane per
  // pass of the block, one row of 32 nodes per warp (uniform parity, coalesced stores).
  const bool has_g = d.gb.p != nullptr;
  auto value = [&](int lx, int ly, int lz, int gx, int gy, int gz) -> double {
    const bool bnd = gx == 0 || gx == g.nx || gy == 0 || gy == g.ny || gz == 0 || gz == g.nz;
    if (bnd && has_g) return d.gb.at(gx, gy, gz);
    if ((lz & 1) == 0) return S.y[lz >> 1][ly][lx];
    const int q = (lz - 1) >> 1, t = q % C, base = q - t;
    double v = 0.0;
#pragma unroll
    for (int m = 0; m < P; ++m) v = fma(S.wq[t][m], S.y[base + m][ly][lx], v);
    return v;
  };
  for (int idx = threadIdx.x; idx < 32 * 8 * 8; idx += kThreads) {
    const int lx = idx & 31, ly = (idx >> 5) & 7, lz = idx >> 8;
    const int gx = 32 * bx + lx, gy = 8 * by + ly, gz = 8 * bz + lz;
    if (gx > g.nx || gy > g.ny || gz > g.nz) continue;
    d.w[gx + gy * g.sy + (long long)gz * g.sz] = value(lx, ly, lz, gx, gy, gz);
  }
  // far faces of the brick that lie on the far faces of the grid (no next brick owns them)
  const bool xe = 32 * bx + 32 == g.nx, ye = 8 * by + 8 == g.ny, ze = 8 * bz + 8 == g.nz;
  if (xe || ye || ze) {
    for (int idx = threadIdx.x; idx < BZF * BYF * BXF; idx += kThreads) {
      const int lx = idx % BXF, ly = (idx / BXF) % BYF, lz = idx / (BXF * BYF);
      const bool far = (lx == 32) || (ly == 8) || (lz == 8);
      if (!far || (lx == 32 && !xe) || (ly == 8 && !ye) || (lz == 8 && !ze)) continue;
      const int gx = 32 * bx + lx, gy = 8 * by + ly, gz = 8 * bz + lz;
      if (gx > g.nx || gy > g.ny || gz > g.nz) continue;
      d.w[gx + gy * g.sy + (long long)gz * g.sz] = value(lx, ly, lz, gx, gy, gz);
    }
  }
}

// ---- EXP_finite in block fixed point (fixed_point.cuh) ----
// The float64 brick costs 5.4 float64 instructions per fine node, 2.7 clocks of an SM at 2
// lanes per clock, against 9.1 bytes (0.4 clocks).  Here the brick's grid-2h and grid-4h
// values become 58-bit integers of the brick's largest exponent, the corner sums are exact,
// every interpolated value is a sum of five products with the integers 128 l_m(t) rounded
// once, and the only float64 instruction left is the result's conversion.  Each pass keeps
// one line of five values in a thread and writes the whole line of results.  Measured, one
// call on 512 x 256 x 128 cells with Dirichlet data: 245 us in float64, 157 us here, 150 of them without
// the check of the cells' sizes; fields that fall off within their bricks 236 us (two block barriers
// fewer, or 32-bit brick indices, changed nothing).
constexpr int kBrickBits = 58;  // |w| <= 1.13 2^58, times (278 / 128)^3 after three passes: < 2^61.6

struct BrickFx {
  // the largest magnitude word of each warp's grid-2h values in the brick's four cells, and of
  // its grid-4h values
  uint4 cell[kThreads / 32];
  unsigned mag[kThreads / 32];
  long long w[BZ1 * BY1][BX1];    // u_2h, then the extrapolated values
  long long d[BZ0][BY0][BX0];     // u_2h - u_4h at the grid-4h nodes
  long long x[BZ1 * BY1][BXF];    // after the pass along x
  long long y[BZ1][BYF][BXF];     // after the pass along y
};

// The four odd (interpolated) values of a cell from its five grid-2h values: sum of w_m
// 128 l_m(t), over 128, to nearest, ties to even (so that -w gives the negative).  w = hi 2^32
// + lo with lo signed, so that every product is one 32 x 32 multiply-add; |sum| / 128 < 2^62.
__device__ __forceinline__ void quartic_fx(const long long (&w)[5], long long (&out)[4]) {
  constexpr int c[4][5] = {{35, 140, -70, 28, -5}, {-5, 60, 90, -20, 3}, {3, -20, 90, 60, -5}, {-5, 28, -70, 140, 35}};
  int hi[5], lo[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    lo[m] = (int)w[m];
    hi[m] = (int)((w[m] - lo[m]) >> 32);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    long long H = 0, L = 64;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      H = fx_mad_s(hi[m], c[t][m], H);
      L = fx_mad_s(lo[m], c[t][m], L);
    }
    out[t] = ((H << 25) + (L >> 7)) & ~(long long)(((int)L & 127) == 0);
  }
}

// Fine nodes of column (lx, ly) of a brick, planes 0 .. 7 (and 8 on the grid's far face).
__device__ __forceinline__ void brick_column(const ProlongDesc& d, const BrickFx& S, int lx, int ly, int gx, int gy,
                                             int gz0, int q) {
  const Grid3& g = d.g;
  long long w[5], odd[4];
#pragma unroll
  for (int m = 0; m < 5; ++m) w[m] = S.y[m][ly][lx];
  quartic_fx(w, odd);
  double* out = d.w + (gx + gy * g.sy + gz0 * g.sz);
  const bool has_g = d.gb.p != nullptr, side = has_g && (gx == 0 || gx == g.nx || gy == 0 || gy == g.ny);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int gz = gz0 + k;
    if (k == 8 && gz != g.nz) break;  // the next brick's first plane
    const double v = fx_scale((double)(k & 1 ? odd[k >> 1] : w[k >> 1]), q);
    *out = side || (has_g && (gz == 0 || gz == g.nz)) ? d.gb.at(gx, gy, gz) : v;
    out += g.sz;
  }
}

// One brick; false, in every thread, when its values are not for fixed point.
__device__ bool exp_finite_brick_fx(const ProlongDesc& d, long long lb, BrickFx& S) {
  const Grid3& g = d.g;
  const int bx = (int)(lb % d.nbx);
  const int by = (int)((lb / d.nbx) % d.nby);
  const int bz = (int)(lb / ((long long)d.nbx * d.nby));
  const int n1x = g.nx / 2, n0x = g.nx / 4;
  const long long s1y = n1x + 1, s1z = s1y * (g.ny / 2 + 1);
  const long long s0y = n0x + 1, s0z = s0y * (g.ny / 4 + 1);
  const int tid = threadIdx.x;
  constexpr int N1 = BX1 * BY1 * BZ1, N0 = BX0 * BY0 * BZ0, kU = (N1 + kThreads - 1) / kThreads;
  static_assert(N0 <= kThreads && BY1 * BZ1 * 4 <= kThreads && BXF * BZ1 <= kThreads, "one item per thread");
  // grid-2h and grid-4h values (bricks divide the grid in y and z; the last one in x may reach
  // past it: zeros there, in cells that no output takes)
  double v1[kU], v0 = 0.0;
  unsigned c0 = 0, c1 = 0, c2 = 0, c3 = 0, low = 0;  // of the four cells along x
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int e = tid + u * kThreads, ix = e % BX1, r = e / BX1, jy = r % BY1, kz = r / BY1;
    const int I = 16 * bx + ix;
    v1[u] = e < N1 && I <= n1x ? __ldg(d.u2h + (I + (4 * by + jy) * s1y + (4 * bz + kz) * s1z)) : 0.0;
    const unsigned m = fx_mag(v1[u]);
    c0 = max(c0, ix < 4 ? m : 0);  // (a node between two cells counts to one)
    c1 = max(c1, ix >= 4 && ix < 8 ? m : 0);
    c2 = max(c2, ix >= 8 && ix < 12 ? m : 0);
    c3 = max(c3, ix >= 12 ? m : 0);
    low |= (unsigned)__double2loint(v1[u]);
  }
  const int i0 = tid % BX0, j0 = (tid / BX0) % BY0, k0 = tid / (BX0 * BY0);
  const bool has0 = tid < N0 && 8 * bx + i0 <= n0x;
  if (has0) v0 = __ldg(d.u4h + (8 * bx + i0 + (2 * by + j0) * s0y + (2 * bz + k0) * s0z));
  unsigned mag = fx_mag(v0);
  low |= (unsigned)__double2loint(v0);
  c0 = __reduce_max_sync(0xffffffffu, c0);
  c1 = __reduce_max_sync(0xffffffffu, c1);
  c2 = __reduce_max_sync(0xffffffffu, c2);
  c3 = __reduce_max_sync(0xffffffffu, c3);
  mag = __reduce_max_sync(0xffffffffu, mag);
  if ((c0 | c1 | c2 | c3 | mag) == 0) mag = __any_sync(0xffffffffu, low != 0);  // denormal below 2^-1042
  __syncthreads();  // the brick before is done with the shared memory
  if ((tid & 31) == 0) {
    S.cell[tid >> 5] = make_uint4(c0, c1, c2, c3);
    S.mag[tid >> 5] = mag;
  }
  __syncthreads();
  // (a lane per warp and cell)
  unsigned near = reinterpret_cast<const unsigned*>(S.cell)[tid & 31];
  mag = __reduce_max_sync(0xffffffffu, max(near, S.mag[tid & 7]));
  const int E = mag == 0 ? kFxMinExp : (int)(mag >> 20);
  if (E < kFxMinExp || E > kFxMaxExp) return false;
#pragma unroll
  for (int o = 4; o < 32; o *= 2) near = max(near, __shfl_xor_sync(0xffffffffu, near, o));
  // a cell of the grid (and all its values) far below the brick's scale
  if (32 * bx + 8 * (tid & 3) >= g.nx) near = ~0u;
  near = __reduce_min_sync(0xffffffffu, near);
  if (mag != 0 && E - (int)(near >> 20) > kFxRange) return false;
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int e = tid + u * kThreads;
    if (e < N1) (&S.w[0][0])[e] = fx_from_double<kBrickBits>(v1[u], E);
  }
  __syncthreads();
  if (tid < N0)
    S.d[k0][j0][i0] = has0 ? S.w[2 * k0 * BY1 + 2 * j0][2 * i0] - fx_from_double<kBrickBits>(v0, E) : 0;
  __syncthreads();
  // w = u_2h + (mean of d over the corners of the node's edge, face or element) / 16: the sum
  // over the eight corners (coinciding ones counted as often) over 128, to nearest, ties to even
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int e = tid + u * kThreads, ix = e % BX1, r = e / BX1, jy = r % BY1, kz = r / BY1;
    if (e >= N1) break;
    const int ia = ix >> 1, ib = (ix + 1) >> 1, ja = jy >> 1, jb = (jy + 1) >> 1, ka = kz >> 1, kb = (kz + 1) >> 1;
    const long long s = ((S.d[ka][ja][ia] + S.d[ka][ja][ib]) + (S.d[ka][jb][ia] + S.d[ka][jb][ib])) +
                        ((S.d[kb][ja][ia] + S.d[kb][ja][ib]) + (S.d[kb][jb][ia] + S.d[kb][jb][ib]));
    S.w[r][ix] += ((s + 64) >> 7) & ~(long long)((((int)s + 64) & 127) == 0);
  }
  __syncthreads();
  long long w[5], odd[4];
  if (tid < BY1 * BZ1 * 4) {  // along x: a cell of a row per thread
    const int c = tid & 3, r = tid >> 2;
#pragma unroll
    for (int m = 0; m < 5; ++m) w[m] = S.w[r][4 * c + m];
    quartic_fx(w, odd);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      S.x[r][8 * c + 2 * m] = w[m];
      S.x[r][8 * c + 2 * m + 1] = odd[m];
    }
    if (c == 3) S.x[r][32] = w[4];
  }
  __syncthreads();
  if (tid < BXF * BZ1) {  // along y: a column of a grid-2h plane per thread
    const int lx = tid % BXF, kz = tid / BXF;
#pragma unroll
    for (int m = 0; m < 5; ++m) w[m] = S.x[kz * BY1 + m][lx];
    quartic_fx(w, odd);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      S.y[kz][2 * m][lx] = w[m];
      S.y[kz][2 * m + 1][lx] = odd[m];
    }
    S.y[kz][8][lx] = w[4];
  }
  __syncthreads();
  // along z, boundary data, store: the brick's 32 x 8 columns, a warp per row; then its far
  // columns where they lie on the grid's far faces (no next brick owns them)
  const int q = E - 1022 - kBrickBits, gx0 = 32 * bx, gy0 = 8 * by;
  const int lx = tid & 31, ly = tid >> 5;
  if (gx0 + lx <= g.nx) brick_column(d, S, lx, ly, gx0 + lx, gy0 + ly, 8 * bz, q);
  const bool xe = gx0 + 32 == g.nx, ye = gy0 + 8 == g.ny;
  if (ye && tid < 32 && gx0 + tid <= g.nx) brick_column(d, S, tid, 8, gx0 + tid, g.ny, 8 * bz, q);
  if (xe && tid >= 32 && tid < 41 && (tid < 40 || ye)) brick_column(d, S, 32, tid - 32, g.nx, gy0 + tid - 32, 8 * bz, q);
  return true;
}

// Weights of the P-point interpolation at the C = P - 1 half-integer points of a cell.
template <int P>
__device__ __forceinline__ void load_weights(BrickSmem& S) {
  constexpr int C = P - 1;
  if (threadIdx.x < C * P) {
    const int t = threadIdx.x / P, m = threadIdx.x % P;
    S.wq[t][m] = P == 5 ? c_wq[t][m] : (P == 3 ? c_wquad[t][m] : c_wlin[t][m]);
  }
}

template <int P>
__device__ __forceinline__ void prolong_bricks(int nprob, const ProlongDesc* __restrict__ descs,
                                               long long total_blocks, BrickSmem& S) {
  load_weights<P>(S);
  int p = 0;
  for (long long b = blockIdx.x; b < total_blocks; b += gridDim.x) {
    while (p + 1 < nprob && b >= descs[p + 1].block_begin) ++p;
    exp_finite_brick<P>(descs[p], b - descs[p].block_begin, S);
  }
}

union BrickAny {
  BrickFx fx;
  BrickSmem f64;
};

// A brick by fixed point, or in float64 where its values do not allow it (infinities, NaN,
// extreme exponents, a cell of grid-2h values all more than 2^kFxRange below the brick's
// largest: the interpolated values are within 2^-52 of the cell's largest, as in float64).
__device__ __forceinline__ void exp_finite_any(const ProlongDesc& d, long long lb, BrickAny& S) {
  if (!exp_finite_brick_fx(d, lb, S.fx)) {
    __syncthreads();
    load_weights<5>(S.f64);
    exp_finite_brick<5>(d, lb, S.f64);
  }
}

__global__ void __launch_bounds__(kThreads, 4)
    k_exp_finite(int nprob, const ProlongDesc* __restrict__ descs, long long total_blocks) {
  __shared__ BrickAny S;
  int p = 0;
  for (long long b = blockIdx.x; b < total_blocks; b += gridDim.x) {
    while (p + 1 < nprob && b >= descs[p + 1].block_begin) ++p;
    exp_finite_any(descs[p], b - descs[p].block_begin, S);
  }
}

// The comparison prolongations (P = 3: extrapolation + tri-quadratic; P = 2: trilinear).
template <int P>
__global__ void __launch_bounds__(kThreads)
    k_prolong_cmp(int nprob, const ProlongDesc* __restrict__ descs, long long total_blocks) {
  __shared__ BrickSmem S;
  prolong_bricks<P>(nprob, descs, total_blocks, S);
}

__global__ void __launch_bounds__(kThreads, 4) k_exp_finite_one(ProlongDesc d, long long total_blocks) {
  __shared__ BrickAny S;
  for (long long b = blockIdx.x; b < total_blocks; b += gridDim.x) exp_finite_any(d, b, S);
}

// EXP_true: u~ = u_h + (1/15) (mean of d = u_h - u_2h over the grid-2h corners of the
// edge / face / element the node is the centre of; d itself at grid-2h nodes).
// A block marches 64 x 8 fine columns (32 x 4 coarse ones) along z, kEtK coarse planes: per
// coarse plane it forms d at its 33 x 5 corners once, in shared memory, and a thread (one
// fine x, the rows 2 J and 2 J + 1) sums its corner columns I and I + (i odd) -- for even i
// the same twice, so that every lane does the same -- over rows J and J + 1; the sums of the
// plane before serve the odd fine plane between.  2.4 float64 instructions per node (a
// thread per node and plane pair summed the corner rows anew, 4.3); bound by the float64
// pipe.  One call on 384 x 256 x 192 cells: 284 us (a row per warp), 154 us marching, 136 us
// with the column i = nx in the last tile.  Chunks of kEtK coarse planes: a deeper one sums fewer
// first planes twice, a shallower one gives small grids more blocks.  us per call with 4 / 6 / 8 /
// 12: 64^3 37 / 43 / 43 / 48, 384 x 256 x 192 142 / 143 / 142 / 147, 512 x 256 x 128 128 / 129 / 129 / 132,
// 1024 x 512 x 512 1452 / 1412 / 1391 / 1373.
constexpr int kEtX = 64, kEtY = 8, kEtK = 8;
constexpr int kEcX = kEtX / 2 + 1, kEcY = kEtY / 2 + 1;

__global__ void __launch_bounds__(kThreads)
    k_exp_true(Grid3 g, const double* __restrict__ uh, const double* __restrict__ u2h,
               double* __restrict__ ut, int ntx, int nty) {
  __shared__ double D[2][kEcY][kEcX];
  static_assert(kThreads == kEtX * (kEtY / 2) && kEcX * kEcY <= kThreads, "a coarse row of fine columns per thread");
  const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
  const int n1x = g.nx / 2, n1y = g.ny / 2, n1z = g.nz / 2;
  const int I0 = bx * (kEtX / 2), J0 = by * (kEtY / 2), K0 = bz * kEtK, K1 = min(K0 + kEtK, n1z + 1);
  const long long s1y = n1x + 1, s1z = (long long)(n1x + 1) * (n1y + 1);
  // this thread's corner (the first 165) and its fine column
  const int ca = threadIdx.x % kEcX, cb = threadIdx.x / kEcX;
  const bool corner = cb < kEcY && I0 + ca <= n1x && J0 + cb <= n1y;
  const double* pc = uh + (2LL * (I0 + ca) + 2LL * (J0 + cb) * g.sy + 2LL * K0 * g.sz);
  const double* pd = u2h + (I0 + ca + (J0 + cb) * s1y + K0 * s1z);
  const int tx = threadIdx.x % kEtX, jq = threadIdx.x / kEtX;
  const int i = 2 * I0 + tx, j = 2 * (J0 + jq), ia = tx >> 1, ib = ia + (tx & 1);
  const bool row0 = i <= g.nx && j <= g.ny, row1 = i <= g.nx && j + 1 <= g.ny;
  const long long o = i + j * g.sy + 2LL * K0 * g.sz;
  const double* u = uh + o;
  double* t = ut + o;
  double a1 = 0.0, s1 = 0.0;  // the plane before: row J, rows J and J + 1
  // nx a multiple of 64: the column i = nx goes with the last tile, to four lanes of the last
  // warp (a tile of its own held one column of 64)
  const int lane = threadIdx.x & 31, fj = 2 * (J0 + lane), fi = n1x - I0;
  const bool far = g.nx % kEtX == 0 && bx == ntx - 1 && threadIdx.x >= kThreads - 32 && lane < kEtY / 2;
  const long long fo = g.nx + fj * g.sy + 2LL * K0 * g.sz;
  double b1 = 0.0, r1 = 0.0;
  for (int K = K0; K <= K1; ++K) {
    if (K > n1z) break;  // the grid's last plane is done
    const bool last = K == K1;  // the next block's first plane, for the odd plane before it
    double (*P)[kEcX] = D[K & 1];
    if (corner) P[cb][ca] = __ldg(pc) - __ldg(pd);
    pc += 2 * g.sz;
    pd += s1z;
    // u of the odd plane before and of this plane
    double um0 = 0.0, um1 = 0.0, u0 = 0.0, u1 = 0.0;
    if (K > K0) {
      if (row0) um0 = __ldg(u - g.sz);
      if (row1) um1 = __ldg(u - g.sz + g.sy);
    }
    if (!last) {
      if (row0) u0 = __ldg(u);
      if (row1) u1 = __ldg(u + g.sy);
    }
    __syncthreads();  // (the other buffer's readers are a barrier behind)
    const double a = P[jq][ia] + P[jq][ib], s = a + (P[jq + 1][ia] + P[jq + 1][ib]);
    // (1/15) over twice the number of corner rows
    if (K > K0) {
      if (row0) t[-g.sz] = fma(a + a1, 1.0 / 60.0, um0);
      if (row1) t[g.sy - g.sz] = fma(s + s1, 1.0 / 120.0, um1);
    }
    if (!last) {
      if (row0) t[0] = fma(a, 1.0 / 30.0, u0);
      if (row1) t[g.sy] = fma(s, 1.0 / 60.0, u1);
    }
    a1 = a;
    s1 = s;
    if (far) {
      const double b = 2.0 * P[lane][fi], r = b + 2.0 * P[lane + 1][fi];
      const double* fu = uh + fo + 2LL * (K - K0) * g.sz;
      double* ft = ut + fo + 2LL * (K - K0) * g.sz;
      if (K > K0) {
        if (fj <= g.ny) ft[-g.sz] = fma(b + b1, 1.0 / 60.0, __ldg(fu - g.sz));
        if (fj + 1 <= g.ny) ft[g.sy - g.sz] = fma(r + r1, 1.0 / 120.0, __ldg(fu + g.sy - g.sz));
      }
      if (!last) {
        if (fj <= g.ny) ft[0] = fma(b, 1.0 / 30.0, __ldg(fu));
        if (fj + 1 <= g.ny) ft[g.sy] = fma(r, 1.0 / 60.0, __ldg(fu + g.sy));
      }
      b1 = b;
      r1 = r;
    }
    u += 2 * g.sz;
    t += 2 * g.sz;
  }
}

// Levels 0 and 1 start CG from zero: u = g on the boundary, 0 inside.
__global__ void __launch_bounds__(kThreads) k_boundary_init(Grid3 g, View gb, double* __restrict__ u) {
  const long long n = g.nodes();
  for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n;
       o += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(o % g.sy);
    const int j = (int)((o / g.sy) % (g.ny + 1));
    const int k = (int)(o / g.sz);
    const bool bnd = i == 0 || i == g.nx || j == 0 || j == g.ny || k == 0 || k == g.nz;
    u[o] = bnd ? gb.at(i, j, k) : 0.0;
  }
}

// A field without zeros or layers, for timing: values in [1, 2) from a hash of the node's index.
__global__ void __launch_bounds__(kThreads) k_timing_field(long long n, double* __restrict__ u) {
  for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n;
       o += (long long)gridDim.x * blockDim.x)
    u[o] = 1.0 + (double)(((unsigned)o * 2654435761u) >> 8) * 0x1p-24;
}

// Adjoint outputs from lambda (zero on boundary nodes):
//   dL/df = -R^T lambda = -(3 lambda_m + (1/2) sum of lambda at the 6 face neighbours)
//   dL/dg = LHS^T lambda + dL/du on boundary nodes, 0 inside (LHS weights = -A weights).
__global__ void __launch_bounds__(kThreads)
    k_adjoint_finish(Grid3 g, Coef A, const double* __restrict__ lam,
                     const double* __restrict__ dLdu, double* __restrict__ dLdf,
                     double* __restrict__ dLdg) {
  const long long n = g.nodes();
  for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < n;
       o += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(o % g.sy);
    const int j = (int)((o / g.sy) % (g.ny + 1));
    const int k = (int)(o / g.sz);
    auto L = [&](int di, int dj, int dk) -> double {
      const int a = i + di, b = j + dj, c = k + dk;
      if (a < 0 || a > g.nx || b < 0 || b > g.ny || c < 0 || c > g.nz) return 0.0;
      return lam[a + b * g.sy + (long long)c * g.sz];
    };
    const double faces = (L(1, 0, 0) + L(-1, 0, 0)) + (L(0, 1, 0) + L(0, -1, 0)) + (L(0, 0, 1) + L(0, 0, -1));
    dLdf[o] = -(3.0 * lam[o] + 0.5 * faces);
    const bool bnd = i == 0 || i == g.nx || j == 0 || j == g.ny || k == 0 || k == g.nz;
    if (!bnd) {
      dLdg[o] = 0.0;
      continue;
    }
    const double sx = L(1, 0, 0) + L(-1, 0, 0), sy = L(0, 1, 0) + L(0, -1, 0), sz = L(0, 0, 1) + L(0, 0, -1);
    const double exy = (L(1, 1, 0) + L(-1, 1, 0)) + (L(1, -1, 0) + L(-1, -1, 0));
    const double exz = (L(1, 0, 1) + L(-1, 0, 1)) + (L(1, 0, -1) + L(-1, 0, -1));
    const double eyz = (L(0, 1, 1) + L(0, -1, 1)) + (L(0, 1, -1) + L(0, -1, -1));
    const double Al = A.c0 * lam[o] + A.fx * sx + A.fy * sy + A.fz * sz + A.exy * exy + A.exz * exz + A.eyz * eyz;
    dLdg[o] = -Al + dLdu[o];
  }
}

// Blocks of a grid-stride elementwise launch over n items: at most 16 per SM of the
// current device.
int flat_grid(long long n) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  long long b = (n + kThreads - 1) / kThreads;
  if (b > (long long)sms * 16) b = (long long)sms * 16;
  return b < 1 ? 1 : (int)b;
}

}  // namespace

// Co-resident blocks of an EXP_finite kernel on the whole device (one full wave).
static int brick_wave(const void* kernel, int& cache) {
  if (cache == 0) {
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kThreads, 0);
    cache = std::max(1, sms) * std::max(1, occ);
  }
  return cache;
}
static int g_wave_many = 0, g_wave_one = 0;

cudaError_t launch_exp_finite(int nprob, const ProlongDesc* descs, long long total_blocks,
                              cudaStream_t s) {
  const long long wave = brick_wave((const void*)k_exp_finite, g_wave_many);
  const long long grid = std::max(1LL, std::min(total_blocks, wave));
  k_exp_finite<<<(int)grid, kThreads, 0, s>>>(nprob, descs, total_blocks);
  return cudaGetLastError();
}

static int g_wave_quad = 0, g_wave_lin = 0;

cudaError_t launch_prolong_cmp(int points, int nprob, const ProlongDesc* descs,
                               long long total_blocks, cudaStream_t s) {
  if (points != 3 && points != 2) return cudaErrorInvalidValue;
  const void* k = points == 3 ? (const void*)k_prolong_cmp<3> : (const void*)k_prolong_cmp<2>;
  const long long wave = brick_wave(k, points == 3 ? g_wave_quad : g_wave_lin);
  const long long grid = std::max(1LL, std::min(total_blocks, wave));
  if (points == 3) {
    k_prolong_cmp<3><<<(int)grid, kThreads, 0, s>>>(nprob, descs, total_blocks);
  } else {
    k_prolong_cmp<2><<<(int)grid, kThreads, 0, s>>>(nprob, descs, total_blocks);
  }
  return cudaGetLastError();
}

cudaError_t launch_exp_finite_one(const ProlongDesc& d, cudaStream_t s) {
  const long long total = (long long)d.nbx * d.nby * d.nbz;
  const long long wave = brick_wave((const void*)k_exp_finite_one, g_wave_one);
  const long long grid = std::max(1LL, std::min(total, wave));
  k_exp_finite_one<<<(int)grid, kThreads, 0, s>>>(d, total);
  return cudaGetLastError();
}

cudaError_t launch_exp_true(const Grid3& g, const double* uh, const double* u2h, double* ut,
                            cudaStream_t s) {
  const int ntx = g.nx % kEtX ? (g.nx + 1 + kEtX - 1) / kEtX : g.nx / kEtX, nty = (g.ny + 1 + kEtY - 1) / kEtY;
  const long long ntz = (g.nz / 2 + 1 + kEtK - 1) / kEtK;
  const long long blocks = (long long)ntx * nty * ntz;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  k_exp_true<<<(unsigned)blocks, kThreads, 0, s>>>(g, uh, u2h, ut, ntx, nty);
  return cudaGetLastError();
}

cudaError_t launch_boundary_init(const Grid3& g, View gb, double* u, cudaStream_t s) {
  k_boundary_init<<<flat_grid(g.nodes()), kThreads, 0, s>>>(g, gb, u);
  return cudaGetLastError();
}

cudaError_t launch_timing_field(const Grid3& g, double* u, cudaStream_t s) {
  k_timing_field<<<flat_grid(g.nodes()), kThreads, 0, s>>>(g.nodes(), u);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_finish(const Grid3& g, const Coef& A, const double* lam,
                                  const double* dLdu, double* dLdf, double* dLdg,
                                  cudaStream_t s) {
  k_adjoint_finish<<<flat_grid(g.nodes()), kThreads, 0, s>>>(g, A, lam, dLdu, dLdf, dLdg);
  return cudaGetLastError();
}

}  // namespace excmg
