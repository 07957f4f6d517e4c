// CUDA kernels of libbssn, templated on the finite-difference order P.
//
// Design. On GB300 the FP64 pipe issues ~74x fewer operations per second
// than the FP32 pipe, so the double-precision forms spend as few FP64
// instructions per grid point as possible:
//
//  * k_derivs (bssn_fixed.cuh): all finite differences, exactly, on the
//    integer pipes, written to a record per tile.
//  * k_algebra (bssn_stage64.cu): one thread per interior point: reads the record, forms the
//    pointwise right-hand side and the RK stage update in double precision.
//
// The constraints and the Weyl scalars still gather their own derivatives in
// double precision (k_diffs, gather). The FP32-RHS form is bssn_stage32.cuh.
#pragma once
#include <type_traits>

#include "bssn_bounds.cuh"
#include "bssn_common.cuh"
#include "bssn_point.cuh"

namespace bssn {

__device__ __forceinline__ double fmaR(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmaR(float a, float b, float c) { return fmaf(a, b, c); }

__device__ __forceinline__ void point_coords(const Layout& L, long long lin, int& i, int& j, int& k) {
  i = (int)(lin % L.nx);
  const long long t = lin / L.nx;
  j = (int)(t % L.ny);
  k = (int)(t / L.ny);
}

// Rows (j, k) visited brick by brick: slabs of BZ planes, each cut into
// bricks of BY rows, rows of a brick z-outer and y-inner (the last slab and
// brick of each axis may be shorter). Maps the position r of a row in that
// order to (j, k). Blocks launched in order then work on a compact region of
// the grid, so the stencil's z-neighbour planes stay in L2.
template <int BY, int BZ>
__device__ __forceinline__ void brick_row(long long r, int ny, int nz, int& j, int& k) {
  const long long slab = (long long)BZ * ny;
  const int kb = (int)(r / slab);
  const long long rr = r - kb * slab;
  const int hz = min(BZ, nz - kb * BZ);
  const int jb = (int)(rr / ((long long)BY * hz));
  const long long rrr = rr - (long long)jb * BY * hz;
  const int hy = min(BY, ny - jb * BY);
  k = kb * BZ + (int)(rrr / hy);
  j = jb * BY + (int)(rrr % hy);
}

// Brick shape (rows x planes) of the traversal of kernels that gather from
// the state and the difference tables.
constexpr int STAGE_BRICK_Y64 = 8, STAGE_BRICK_Z64 = 32;

// ------------------------------------------------------------------ differences
template <int P, typename R>
__global__ void __launch_bounds__(256) k_diffs(Layout L, const R* __restrict__ u, R* __restrict__ dX,
                                               R* __restrict__ dY) {
  constexpr int H = FD<P>::H;
  const long long ex = L.nx, ey = L.ny + 2 * H, ez = L.nz + 2 * H;
  const long long lin = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (lin >= ex * ey * ez) return;
  const int i = (int)(lin % ex);
  const long long t = lin / ex;
  const int j = (int)(t % ey) - H;
  const int k = (int)(t / ey) - H;
  const long long p = L.off0 + i + j * L.sy + k * L.sz;
  const bool doy = (j >= 0 && j < L.ny);
  if (!in_range(p - H * L.sy, p + H * L.sy, padded_points(L))) return;
#pragma unroll 1
  for (int m = 0; m < NM; ++m) {
    const R* v = u + mvar(m) * L.vs;
#pragma unroll
    for (int a = 1; a <= H; ++a) {
      const long long o = (long long)(m * H + a - 1) * L.vs + p;
      dX[o] = __ldg(v + p + a) - __ldg(v + p - a);
      if (doy) dY[o] = __ldg(v + p + a * L.sy) - __ldg(v + p - a * L.sy);
    }
  }
}

// first derivative along a stride from the state: sum_a c_a (u_a - u_-a)
template <int H, typename R>
__device__ __forceinline__ R d1_direct(const R* __restrict__ v, long long p, long long s, const R* c) {
  R r = c[1] * (__ldg(v + p + s) - __ldg(v + p - s));
#pragma unroll
  for (int a = 2; a <= H; ++a) r = fmaR(c[a], __ldg(v + p + a * s) - __ldg(v + p - a * s), r);
  return r;
}

// first derivative from a difference table: sum_a c_a tab_a
template <int H, typename R>
__device__ __forceinline__ R d1_table(const R* __restrict__ tab, long long vs, long long p, const R* c) {
  R r = c[1] * __ldg(tab + p);
#pragma unroll
  for (int a = 2; a <= H; ++a) r = fmaR(c[a], __ldg(tab + (a - 1) * vs + p), r);
  return r;
}

// mixed derivative: sum_a sum_b cm_ab (tab_a(p + b s) - tab_a(p - b s))
template <int H, typename R>
__device__ __forceinline__ R dmix_table(const R* __restrict__ tab, long long vs, long long p, long long s,
                                        const R (*cm)[5]) {
  R r = R(0);
#pragma unroll
  for (int a = 1; a <= H; ++a) {
    const R* t = tab + (a - 1) * vs;
#pragma unroll
    for (int b = 1; b <= H; ++b) r = fmaR(cm[a][b], __ldg(t + p + b * s) - __ldg(t + p - b * s), r);
  }
  return r;
}

// Gather every derivative of the constraints and Weyl scalars at point p.
// With NMIX < NM only the first NMIX variables with second derivatives get
// their derivatives (7: W and gt_ij, all the Hamiltonian constraint needs);
// the lapse's and shift's are then left zero.
template <int P, typename R, int NMIX = NM>
__device__ __forceinline__ void gather(const Layout& L, const Coef<R>& C, const R* __restrict__ u,
                                       const R* __restrict__ dX, const R* __restrict__ dY, long long p,
                                       PointIn<R>& Q) {
  constexpr int H = FD<P>::H;
  const long long vs = L.vs;
  const long long st[3] = {1, L.sy, L.sz};
#pragma unroll
  for (int v = 0; v < NV; ++v) Q.u[v] = __ldg(u + v * vs + p);
  if (NMIX < NM) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      Q.da[d] = R(0);
#pragma unroll
      for (int i = 0; i < 3; ++i) Q.db[d][i] = R(0);
    }
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      Q.dda[s] = R(0);
#pragma unroll
      for (int i = 0; i < 3; ++i) Q.ddb[i][s] = R(0);
    }
  }

  // ---- the 11 variables with second derivatives
#pragma unroll 1
  for (int m = 0; m < NMIX; ++m) {
    const int var = mvar(m);
    const R* v = u + var * vs;
    const R* tx = dX + (long long)m * H * vs;
    const R* ty = dY + (long long)m * H * vs;
    R d1v[3], d2v[6];
    d1v[0] = d1_table<H>(tx, vs, p, C.c1[0]);
    d1v[1] = d1_table<H>(ty, vs, p, C.c1[1]);
    d1v[2] = d1_direct<H>(v, p, L.sz, C.c1[2]);
    const R m2u0 = R(-2) * __ldg(v + p);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      R dd = R(0);
#pragma unroll
      for (int a = 1; a <= H; ++a) {
        const R sa = (__ldg(v + p + a * st[d]) + __ldg(v + p - a * st[d])) + m2u0;
        dd = fmaR(C.c2[d][a], sa, dd);
      }
      d2v[sym(d, d)] = dd;
    }
    d2v[1] = dmix_table<H>(tx, vs, p, L.sy, C.cm[0]);  // xy
    d2v[2] = dmix_table<H>(tx, vs, p, L.sz, C.cm[1]);  // xz
    d2v[4] = dmix_table<H>(ty, vs, p, L.sz, C.cm[2]);  // yz
    if (m == 0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) Q.dW[d] = d1v[d];
#pragma unroll
      for (int s = 0; s < 6; ++s) Q.ddW[s] = d2v[s];
    } else if (m <= 6) {
#pragma unroll
      for (int d = 0; d < 3; ++d) Q.dg[d][m - 1] = d1v[d];
#pragma unroll
      for (int s = 0; s < 6; ++s) Q.ddg[m - 1][s] = d2v[s];
    } else if (m == 7) {
#pragma unroll
      for (int d = 0; d < 3; ++d) Q.da[d] = d1v[d];
#pragma unroll
      for (int s = 0; s < 6; ++s) Q.dda[s] = d2v[s];
    } else {
#pragma unroll
      for (int d = 0; d < 3; ++d) Q.db[d][m - 8] = d1v[d];
#pragma unroll
      for (int s = 0; s < 6; ++s) Q.ddb[m - 8][s] = d2v[s];
    }
  }

  // ---- first derivatives of K and Gt^i
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Q.dK[d] = d1_direct<H>(u + V_TRK * vs, p, st[d], C.c1[d]);
#pragma unroll
    for (int i = 0; i < 3; ++i) Q.dGam[d][i] = d1_direct<H>(u + (V_GAM1 + i) * vs, p, st[d], C.c1[d]);
  }
}

// Resident blocks per SM asked of the compiler for the kernels that gather
// in double precision: warps hide load latency better than registers do.
constexpr int STAGE_F64_MIN_BLOCKS = 4;

// ------------------------------------------------------------------ dissipation only
template <int P, typename R>
__global__ void __launch_bounds__(256) k_ko(Layout L, Coef<R> C, const double* __restrict__ u, double* rhs) {
  using F = FD<P>;
  const long long lin = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (lin >= L.npts) return;
  int i, j, k;
  point_coords(L, lin, i, j, k);
  const long long p = L.off0 + i + j * L.sy + k * L.sz;
  const long long st[3] = {1, L.sy, L.sz};
#pragma unroll 1
  for (int var = 0; var < NV; ++var) {
    const double* v = u + var * L.vs;
    const R m2u0 = R(-2) * (R)__ldg(v + p);
    R ko = R(0);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int a = 1; a <= F::R; ++a)
        ko = fmaR(C.ko[d][a], ((R)__ldg(v + p + a * st[d]) + (R)__ldg(v + p - a * st[d])) + m2u0, ko);
    rhs[var * L.vs + p] += (double)ko;
  }
}

// ------------------------------------------------------------------ constraints
// Per-block partial results: 7 sums of squares, 7 maxima, written to
// part[blockIdx.x * 14 + q]. Always double precision. With HONLY the
// Hamiltonian constraint alone (the momentum and Gamma slots stay 0, and
// the derivatives only they need are not formed); its values are the same
// bits as in the full evaluation.
template <int P, bool HONLY>
__global__ void __launch_bounds__(128, STAGE_F64_MIN_BLOCKS) k_constraints(Layout L, Coef<double> C, const double* __restrict__ u,
                                                     const double* __restrict__ dX, const double* __restrict__ dY,
                                                     double* ham, double* mom, double* gcon, double* part,
                                                     unsigned int* flag) {
  constexpr int H = FD<P>::H;
  const long long lin = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double c[7];
#pragma unroll
  for (int q = 0; q < 7; ++q) c[q] = 0.0;
  bool bad = false;
  int i = 0, j = 0, k = 0;
  long long p = 0;
  if (lin < L.npts) {
    i = (int)(lin % L.nx);
    brick_row<STAGE_BRICK_Y64, STAGE_BRICK_Z64>(lin / L.nx, L.ny, L.nz, j, k);  // rows in brick order, as k_stage
    p = L.off0 + i + j * L.sy + k * L.sz;
  }
  // no early return here: every thread takes part in the block reduction
  if (lin < L.npts && in_range(p - FD<P>::R * L.sz, p + FD<P>::R * L.sz, padded_points(L))) {
    PointIn<double> Q;
    gather<P, double, HONLY ? 7 : NM>(L, C, u, dX, dY, p, Q);
    double dAt[3][6];
    const long long st[3] = {1, L.sy, L.sz};
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int s = 0; s < 6; ++s) dAt[d][s] = HONLY ? 0.0 : d1_direct<H>(u + (V_AT11 + s) * L.vs, p, st[d], C.c1[d]);
    const double iW = 1.0 / Q.u[V_W];
    constraints_point<double>(Q, dAt, iW, c);
    if (HONLY)
#pragma unroll
      for (int q = 1; q < 7; ++q) c[q] = 0.0;
    if (ham) ham[p] = c[0];
    if (mom && !HONLY)
#pragma unroll
      for (int a = 0; a < 3; ++a) mom[a * L.vs + p] = c[1 + a];
    if (gcon && !HONLY)
#pragma unroll
      for (int a = 0; a < 3; ++a) gcon[a * L.vs + p] = c[4 + a];
#pragma unroll
    for (int q = 0; q < 7; ++q) bad |= !isfinite(c[q]);
    bad |= !(Q.u[V_W] > 0.0);  // the conformal factor must stay positive
  }
  if (bad) atomicOr(flag, 1u);
  __shared__ double red[4][14];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    double s = c[q] * c[q];
    double m = fabs(c[q]);
    if (!(m == m)) m = 0.0;  // NaN handled by the flag
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_down_sync(0xffffffffu, s, o);
      m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    }
    if (lane == 0) {
      red[warp][q] = s;
      red[warp][7 + q] = m;
    }
  }
  __syncthreads();
  if (threadIdx.x < 14) {
    const int q = threadIdx.x;
    double r = red[0][q];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = (q < 7) ? r + red[w][q] : fmax(r, red[w][q]);
    part[(long long)blockIdx.x * 14 + q] = r;
  }
}

}  // namespace bssn
