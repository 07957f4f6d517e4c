// FP64 derivatives on the integer pipes.
//
// GB300 issues FP64 at 1.68 operations per clock and SM, 32-bit integer
// operations at up to 128. The finite-difference stencils are sums of stored
// values with small rational weights, so they are evaluated here exactly, in
// fixed point, and rounded to double once:
//
//  * one block takes one variable on one tile of 8 x 8 x 8 interior points
//    with its halo. 2^E is the power of two above the largest value of the
//    tile and its halo, and every value becomes the integer
//    n = trunc(u 2^(59-E)), |n| < 2^59: six bits more than a double's
//    significand has. Values within 2^-6 of 2^E are held exactly, smaller ones
//    to 2^(E-59).
//  * that is enough for a derivative whose own stencil reads some value of at
//    least 2^(E-7): 2^(E-59) is then no more than that value's last bit, which a
//    difference of two such values is rounded to in double precision. Where a
//    point has others (beside a spike or a steep front of the tile, or along a
//    line or in a plane on which the variable is nearly zero: 1 to 3 % of the
//    points of evolved puncture data, in 5 to 15 % of the tiles), what the
//    integers leave out of the tile's values is kept as single-precision
//    fractions of their unit, and the same stencils of those are added
//    (fx_refine). What is coarser still (values of 2^(E-28), 24 bits of the
//    fractions), and all of a tile whose values are not all finite, or so large
//    or small that the scaling could leave the range of doubles, is made from
//    the doubles (fx_fallback): infinities and NaNs then reach exactly the
//    points whose stencils touch them. What a derivative is good to depends on
//    what its stencil reads, and not on what else its tile holds.
//  * n is kept as two limbs, n = hi 2^30 + lo with 0 <= lo < 2^30, so that
//    differences a - b and paired sums a + b - 2c of limbs fit 32 bits and a
//    weighted sum is one 32 x 32 + 64 bit multiply-add per limb. The weights
//    are the integers of the stencils over a common denominator.
//  * mixed derivatives apply the first-derivative weights along y or z to
//    the exact first-derivative sums along x or y (three limbs, in shared
//    memory).
//  * the sum is rounded to the nearest double; the algebra (or, where h differs
//    by axis, this kernel) scales it by 1/(denominator h).
//
// Apart from that of the paired sums (fx_pair) no rounding happens before, so
// a constant field has exactly zero derivatives and the result does not
// depend on the order of the terms.
//
// k_derivs writes the derivatives to a record, one slot per tile
// (rec[(slot * nout + output) * vol + point of the tile]); the algebra kernel
// reads them back. At 128^3, 8th order, one stage took 17.26 ms (+ 0.40 ms of
// difference tables) when one kernel did stencils and algebra on the FP64
// pipe (4375 FP64 instructions per point), 6.4 ms this way (938). Against a
// quadruple-precision evaluation the right-hand side's error is no larger than
// before in any variable, and 1e-16 instead of 1e-14 for W, gt_ii and alpha.
// Looking after coarse derivatives costs 3 % of an RK4 step of evolved punctures
// at 128^3 (25.5 -> 26.2 ms) and of a small hierarchy's (17.6 -> 18.2), 5 % of an
// RK3 step at 100^3, 9 % of a step of 192 patches whose tiles have such points in
// one case of five (378 -> 412); from the doubles alone, 18 % at 128^3, 57 % at
// 100^3. On a grid with points on a symmetry plane, where variables are the
// rounding of zero, the doubles serve that plane (101^3: 10.0 -> 11.9 ms).
#pragma once
#include <cmath>
#include <type_traits>

#include "bssn_bounds.cuh"
#include "bssn_common.cuh"

namespace bssn {

constexpr int FX_T = 8;          // tile edge
constexpr int FX_THREADS = 512;  // threads of k_derivs: one tile point each

// Integer weights: first derivative W1/D1, second derivative W2/D1^2, paired
// form of the upwinded first derivative
//   sum_i UP[i] u(s o_i) = [ sum_a WT[a] (u_sa - u_-sa) + SK Delta ] / DU,
// Delta = sum_a WK[a] (u_a + u_-a - 2 u_0) the 2r-th difference that is also
// the Kreiss-Oliger operator (the even part of the upwinded stencil has to
// vanish on all even powers below 2r, which leaves only this one), s = +-1.
template <int P> struct FX;
template <> struct FX<4> {
  static constexpr int D1 = 12, DU = 24, SK = 1;
  static __host__ __device__ constexpr int W1(int a) { return a == 1 ? 8 : -1; }
  static __host__ __device__ constexpr int W2(int a) { return a == 1 ? 192 : -12; }
  static __host__ __device__ constexpr int WT(int a) { return a == 1 ? 21 : (a == 2 ? -6 : 1); }
  static __host__ __device__ constexpr int WK(int a) { return a == 1 ? 15 : (a == 2 ? -6 : 1); }
};
template <> struct FX<8> {
  static constexpr int D1 = 840, DU = 1680, SK = 3;
  static __host__ __device__ constexpr int W1(int a) { return a == 1 ? 672 : (a == 2 ? -168 : (a == 3 ? 32 : -3)); }
  static __host__ __device__ constexpr int W2(int a) {
    return 140 * (a == 1 ? 8064 : (a == 2 ? -1008 : (a == 3 ? 128 : -9)));
  }
  static __host__ __device__ constexpr int WT(int a) {
    return a == 1 ? 1470 : (a == 2 ? -480 : (a == 3 ? 145 : (a == 4 ? -30 : 3)));
  }
  static __host__ __device__ constexpr int WK(int a) {
    return a == 1 ? 210 : (a == 2 ? -120 : (a == 3 ? 45 : (a == 4 ? -10 : 1)));
  }
};

// The record of one point: which derivatives of which variables, and where.
struct DerivList {
  int n, nout;
  signed char var[NV];
  short d1[NV];   // first of 3 outputs (x, y, z), or -1
  short d2[NV];   // first of 6 outputs (xx, xy, xz, yy, yz, zz), or -1
  short ext[NV];  // advection + dissipation, or -1
  signed char s1[NV], s2[NV];  // binary exponents added to the first and second derivatives (0 or -1)

  void add(int v, int o1, int o2, int oe) {
    const bool gt = v >= V_GT11 && v <= V_GT33, gam = v >= V_GAM1 && v <= V_GAM3;
    var[n] = (signed char)v;
    d1[n] = (short)o1;
    d2[n] = (short)o2;
    ext[n] = (short)oe;
    s1[n] = gt || gam ? -1 : 0;  // the algebra takes half of these (Point64)
    s2[n] = gt ? -1 : 0;
    ++n;
  }
};

// Right-hand side: W, gt, alpha, beta (9 outputs each), K and Gt^i (3 each),
// then the 24 advection + dissipation sums.
constexpr int REC_K = 9 * NM, REC_GAM = REC_K + 3, REC_EXT = REC_GAM + 9, REC_RHS = REC_EXT + NV;

// Constraints and Weyl scalars: W and gt (9 each), Gt^i (3 each), all that the
// Hamiltonian constraint and the conformal Ricci tensor need.
constexpr int REC_C_GAM = 9 * 7, REC_HAM = REC_C_GAM + 9;

inline DerivList ham_list() {
  DerivList D{};
  for (int m = 0; m < 7; ++m) D.add(m, 9 * m, 9 * m + 3, -1);
  for (int i = 0; i < 3; ++i) D.add(V_GAM1 + i, REC_C_GAM + 3 * i, -1, -1);
  D.nout = REC_HAM;
  return D;
}

inline DerivList rhs_list() {
  DerivList D{};
  for (int m = 0; m < NM; ++m) D.add(mvar(m), 9 * m, 9 * m + 3, REC_EXT + mvar(m));
  for (int v = 0; v < NV; ++v) {
    if (mixed_index(v) >= 0) continue;
    D.add(v, v == V_TRK ? REC_K : (v >= V_GAM1 && v <= V_GAM3 ? REC_GAM + 3 * (v - V_GAM1) : -1), -1, REC_EXT + v);
  }
  D.nout = REC_RHS;
  return D;
}

// Scales of one grid's stencils. Where h is the same along all axes (cubic)
// the record holds the derivatives' integer sums unscaled, 1/c1 times a first
// and 1/c1^2 times a second derivative (second-derivative weights are brought
// to the denominator D1^2), and the algebra, homogeneous in them, applies c1
// and c1^2 once (a and a2); the dissipation of the three axes is one exact
// sum. Otherwise k_derivs scales every derivative and the algebra's factors
// are 1.
struct FxCoef {
  double c1[3];  // 1 / (D1 h_d)
  double c2[6];  // 1 / (D1^2 h h'), packed as sym()
  double cu[3];  // 1 / (DU h_d)
  double ck[3];  // eps KOSCALE / h_d
  double a, a2;  // what the algebra multiplies first and second derivatives by
  double ia;     // 1 / a
  double b;      // a2 / a: a times this is closer to a2 than a times a
  int cubic;
  int weak;      // little or no dissipation
};

// 1 / (k h h2) to the last bit: what is off here is off by the same part at
// every point.
inline double fx_inverse(double k, double h, double h2 = 1.0) {
  const double p = k * h, pe = std::fma(k, h, -p);
  const double x = p * h2, xe = std::fma(pe, h2, std::fma(p, h2, -x));
  const double q = 1.0 / x;
  return std::fma(q, std::fma(-q, xe, std::fma(-q, x, 1.0)), q);
}

template <int P>
FxCoef make_fx(const bssn_grid_t& G, double eps) {
  using X = FX<P>;
  FxCoef C;
  const double h[3] = {G.dx, G.dy, G.dz};
  for (int d = 0; d < 3; ++d) {
    C.c1[d] = fx_inverse(X::D1, h[d]);
    C.cu[d] = fx_inverse(X::DU, h[d]);
    C.ck[d] = eps * FD<P>::KOSCALE / h[d];
  }
  for (int s = 0; s < 6; ++s) {
    const int i = sym_i(s), j = sym_j(s);
    C.c2[s] = fx_inverse((double)X::D1 * X::D1, h[i], h[j]);
  }
  C.cubic = G.dx == G.dy && G.dy == G.dz;
  C.weak = eps < 0.05;
  C.a = C.cubic ? C.c1[0] : 1.0;
  C.a2 = C.cubic ? C.c2[0] : 1.0;
  C.ia = C.cubic ? X::D1 * h[0] : 1.0;
  const double p = X::D1 * h[0], off = std::fma(-C.a, std::fma((double)X::D1, h[0], -p), std::fma(-C.a, p, 1.0));
  C.b = C.cubic ? std::fma(C.a, 2.0 * off, C.a) : 1.0;
  return C;
}

// Tiles of one grid: extents of a (full) tile, counts, slot volume.
struct FxTiles {
  int tx, ty, tz, ntx, nty, ntz, vol;
};
__host__ __device__ inline FxTiles fx_tiles(int nx, int ny, int nz) {
  FxTiles T;
  T.tx = nx < FX_T ? nx : FX_T;
  T.ty = ny < FX_T ? ny : FX_T;
  T.tz = nz < FX_T ? nz : FX_T;
  T.ntx = (nx + FX_T - 1) / FX_T;
  T.nty = (ny + FX_T - 1) / FX_T;
  T.ntz = (nz + FX_T - 1) / FX_T;
  T.vol = T.tx * T.ty * T.tz;
  return T;
}

// ------------------------------------------------------------------ fixed point
// shifts that give 0 for counts of 64 and more (the PTX rule)
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long x, int n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}
__device__ __forceinline__ unsigned long long fx_shl(unsigned long long x, int n) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}

constexpr int FX_LIMB = 30;
constexpr unsigned int FX_MASK = (1u << FX_LIMB) - 1;
constexpr int FX_HELD = 1 << 22;  // high limb of a value of 2^(E-7)
constexpr int FX_FINE = 2;        // of a value of 2^(E-28), of which fx_rest adds enough

// limbs (lo, hi) of trunc(u 2^(1081 - emax)), emax the largest biased exponent
__device__ __forceinline__ int2 fx_from_double(double u, int emax) {
  const int h = __double2hiint(u);
  const unsigned int l = (unsigned int)__double2loint(u);
  const int ex = (h >> 20) & 0x7ff;
  // (the leading one is wrong for subnormals and zero, which end up 0 all the
  // same: emax is 160 at least)
  const unsigned int mh = ((unsigned int)h & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)__funnelshift_l(l, mh, 6) << 32) | (l << 6);
  const unsigned long long s = (unsigned long long)(long long)(h >> 31);
  const long long n = (long long)((fx_shr(m, emax - ex) ^ s) - s);
  return make_int2((int)((unsigned int)n & FX_MASK), (int)(n >> FX_LIMB));
}

// What fx_from_double leaves out: u 2^(1081 - emax) - n, in (-1, 1), to 2^-32
__device__ __forceinline__ float fx_rest(double u, int emax) {
  const int h = __double2hiint(u);
  const unsigned int l = (unsigned int)__double2loint(u);
  const int sh = emax - ((h >> 20) & 0x7ff);
  const unsigned int mh = ((unsigned int)h & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)__funnelshift_l(l, mh, 6) << 32) | (l << 6);
  const float r = __uint2float_rn((unsigned int)((fx_shl(m, 64 - sh) | fx_shr(m, sh - 64)) >> 32)) * 0x1p-32f;
  return h < 0 ? -r : r;
}

// The sum of two values, rounded to 53 significant bits (ties to even) as a
// double-precision addition rounds it; lo may come out as 2^30. The sums of
// second derivatives keep this one rounding of the double-precision form: on
// data that varies along one axis only, its effect on the derivative along
// that axis (2^-53 |u| / h^2) is larger than any other rounding of the
// right-hand side, and results stay comparable with that form's.
__device__ __forceinline__ int2 fx_pair(int2 p, int2 m) {
  unsigned int lo = (unsigned int)(p.x + m.x);
  const int hi = p.y + m.y + (int)(lo >> FX_LIMB);
  lo &= FX_MASK;
  const int g = max(0, 9 - __clz(hi ^ (hi >> 31)));  // bits of the sum beyond 53
  const unsigned int mk = (1u << g) - 1u;
  lo = (lo + (mk >> 1) + ((lo >> g) & mk & 1u)) & ~mk;
  return make_int2((int)lo, hi);
}

// (hi 2^30 + lo) 2^(emax - 1081), rounded to nearest (ties away from zero)
__device__ __forceinline__ double fx_to_double(long long hi, long long lo, int emax) {
  const long long t = hi + (lo >> FX_LIMB);
  // 96 bits w2:w1:w0, the value times four; magnitude by conditional negation
  unsigned int w0 = (unsigned int)lo << (32 - FX_LIMB), w1 = (unsigned int)t, w2 = (unsigned int)(t >> 32);
  const unsigned int x = (unsigned int)((int)w2 >> 31);
  w0 ^= x;
  w1 ^= x;
  w2 ^= x;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+r"(w0), "+r"(w1), "+r"(w2)
      : "r"(x));
  // the top 64 bits, leading one at bit 63
  const bool p2 = w2 != 0u, p1 = w1 != 0u;
  const unsigned int wa = p2 ? w2 : (p1 ? w1 : w0), wb = p2 ? w1 : (p1 ? w0 : 0u), wc = p2 ? w0 : 0u;
  const int s = __clz((int)wa);
  const unsigned int y1 = __funnelshift_l(wb, wa, s), y0 = __funnelshift_l(wc, wb, s);
  const int e = emax + 34 - s - (p2 ? 0 : (p1 ? 32 : 64));
  unsigned int ml = __funnelshift_r(y0, y1, 11), mh = (y1 >> 11) + ((unsigned int)e << 20) + (x << 31);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(ml), "+r"(mh) : "r"((y0 >> 10) & 1u));
  return __hiloint2double(y1 ? (int)mh : 0, (int)ml);
}

// ------------------------------------------------------------------ double-precision stencils
// Which derivatives of a point: the first and second along axis d (FX_AXIS << d),
// the mixed ones (FX_MIXED for xy, then xz, yz), the axis' share of advection
// and dissipation (FX_EXT << d).
constexpr int FX_AXIS = 1, FX_MIXED = 8, FX_EXT = 64, FX_ALL = 511;
constexpr int FX_BEYOND = 9;  // those shifted by this: too coarse for fx_refine as well

// The derivatives `which` of a point that fixed point does not hold. v: the
// variable, p: the point; has1, has2, hase: which of them the variable's record
// has, half1 and half2: whether it has half the first and second ones. oe holds
// the sum of the other axes unless `which` is FX_ALL. beta: the shift's first
// component at the point, the others vs apart; ko: whether there is a
// dissipation, whose stencil reads further than the upwinded one. Each axis' values are
// loaded before any is used: what these points cost is mostly that latency.
template <int P>
__device__ __noinline__ void fx_fallback(const double* __restrict__ v, long long p, long long sy, long long sz,
                                         const FxCoef& C, const double* __restrict__ beta, long long vs, bool adv,
                                         bool ko, int which, bool has1, bool has2, bool hase, bool half1, bool half2,
                                         double* __restrict__ o1, double* __restrict__ o2, double* __restrict__ oe,
                                         int vol) {
  using F = FD<P>;
  using X = FX<P>;
  constexpr int H = F::H, R = F::R;
  const double f1 = half1 ? 0.5 : 1.0, f2 = half2 ? 0.5 : 1.0;
  v += p;
  const double u0 = v[0], m2 = -2.0 * u0;
  const bool wante = hase && which >= FX_EXT;
  double ext = wante && which != FX_ALL ? *oe : 0.0;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const bool axis = which & (FX_AXIS << d), share = hase && (which & (FX_EXT << d));
    if (!axis && !share) continue;
    const long long st = d == 0 ? 1 : (d == 1 ? sy : sz);
    double up[R + 1], um[R + 1];
#pragma unroll
    for (int a = 1; a <= R; ++a) {
      up[a] = um[a] = 0.0;
      if (a <= H || share) {
        up[a] = v[a * st];
        um[a] = v[-a * st];
      }
    }
    if (axis) {
      double r1 = 0.0, r2 = 0.0;
#pragma unroll
      for (int a = 1; a <= H; ++a) {
        r1 += X::W1(a) * (up[a] - um[a]);
        if (has2) r2 += X::W2(a) * ((up[a] + um[a]) + m2);
      }
      if (has1) o1[d * vol] = f1 * (C.cubic ? r1 : C.c1[d] * r1);
      if (has2) o2[sym(d, d) * vol] = f2 * (C.cubic ? r2 : C.c2[sym(d, d)] * r2);
    }
    if (share) {
      if (ko) {
        double k = 0.0;
#pragma unroll
        for (int a = 1; a <= R; ++a) k += X::WK(a) * ((up[a] + um[a]) + m2);
        ext += C.ck[d] * k;
      }
      if (adv) {
        // the one-sided stencil the sign of beta selects, and no other point
        const double bd = beta[d * vs];
        const bool neg = bd < 0.0;
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < F::UPN; ++i) {
          const int o = F::UPLO + i, b = o < 0 ? -o : o;
          int w = 0;
          if (o == 0)
            for (int a = 1; a <= R; ++a) w -= 2 * X::SK * X::WK(a);
          else
            w = X::SK * X::WK(b) + (o > 0 ? X::WT(o) : -X::WT(-o));
          t += w * (o == 0 ? u0 : ((o < 0) != neg ? um[b] : up[b]));
        }
        ext += C.cu[d] * fabs(bd) * t;
      }
    }
  }
  if (wante) *oe = ext;
  if (!has2) return;
  int pair = FX_MIXED;
#pragma unroll 1
  for (int q = 0; q < 3; ++q, pair <<= 1) {
    if (!(which & pair)) continue;
    const long long si = q < 2 ? 1 : sy, sj = q == 0 ? sy : sz;
    double r = 0.0;
#pragma unroll 1
    for (int a = 1; a <= H; ++a) {
      const double *vp = v + a * si, *vm = v - a * si;
      double t = 0.0;
#pragma unroll
      for (int b = 1; b <= H; ++b) t += X::W1(b) * ((vp[b * sj] - vm[b * sj]) - (vp[-b * sj] - vm[-b * sj]));
      r += X::W1(a) * t;
    }
    const int c = q == 2 ? 4 : q + 1;  // packed xy, xz, yz
    o2[c * vol] = f2 * (C.cubic ? r : C.c2[c] * r);
  }
}

// ------------------------------------------------------------------ one tile of one variable
template <int P>
struct FxSmem {
  static constexpr int H = FD<P>::H, R = FD<P>::R;
  static constexpr int BX = FX_T + 2 * R;          // box edge
  static constexpr int EH = FX_T + 2 * H;
  static constexpr int BOX = BX * BX * BX;
  static constexpr int GN = EH * FX_T * FX_T;      // entries of one first-derivative table
  static constexpr size_t bytes = sizeof(int2) * BOX + 3 * sizeof(int4) * GN;
};

// x 2^(emax - 1081) by moving the fields (0 where x is subnormal)
__device__ __forceinline__ double fx_scaled(float x, int emax) {
  const unsigned int b = __float_as_uint(x), m = b & 0x7fffffu;
  const int e = (int)((b >> 23) & 0xff);
  const int hi = (int)((b & 0x80000000u) | (unsigned int)(e + (emax - 185)) << 20 | m >> 3);
  return e ? __hiloint2double(hi, (int)(m << 29)) : 0.0;
}

// Adds to the derivatives `which` of a point what the integers left out of the
// values that its stencils read (r: fx_rest of the point's, in a box like the
// integers'). That is less than one unit a value, so single precision brings a
// sum to 2^-24 of a unit and a derivative to what its own stencil's doubles
// allow. Added in memory, where the point's thread has just written the rest and
// no other adds (a reduction at the L2, with no load to wait for and no FP64
// operation here: 423 -> 412 ms per step of 192 uneven patches).
// The FP64 pipe is the algebra's, so what can be done without it is (192
// uneven patches, a fifth of the tiles with such points: 427 -> 412 ms per step).
template <int P>
__device__ __noinline__ void fx_refine(const float* __restrict__ r, const FxCoef& C, const double* __restrict__ beta,
                                       long long vs, bool adv, int which, bool has1, bool has2, int emax, int emax1,
                                       int emax2, double* __restrict__ o1, double* __restrict__ o2,
                                       double* __restrict__ oe, int vol) {
  using F = FD<P>;
  using X = FX<P>;
  constexpr int H = F::H, R = F::R, BX = FxSmem<P>::BX;
  const float r0 = r[0];
  double ext = 0.0;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    if (!(which & ((FX_AXIS | FX_EXT) << d))) continue;
    const int st = d == 0 ? 1 : (d == 1 ? BX : BX * BX);
    float c1 = 0.f, c2 = 0.f, k = 0.f, t = 0.f;
#pragma unroll
    for (int a = 1; a <= R; ++a) {
      const float p = r[a * st], m = r[-a * st], df = p - m, s = p + m - 2.f * r0;
      if (a <= H) {
        c1 = fmaf((float)X::W1(a), df, c1);
        c2 = fmaf((float)X::W2(a), s, c2);
      }
      k = fmaf((float)X::WK(a), s, k);
      t = fmaf((float)X::WT(a), df, t);
    }
    if (which & (FX_AXIS << d)) {
      const double r1 = fx_scaled(c1, emax1), r2 = fx_scaled(c2, emax2);
      if (has1) atomicAdd(o1 + d * vol, C.cubic ? r1 : C.c1[d] * r1);
      if (has2) atomicAdd(o2 + sym(d, d) * vol, C.cubic ? r2 : C.c2[sym(d, d)] * r2);
    }
    if (which & (FX_EXT << d)) {
      ext = fma(C.ck[d], fx_scaled(k, emax), ext);
      if (adv) {
        const double b = beta[d * vs];
        const float sk = __double2hiint(b) < 0 ? -(float)X::SK : (float)X::SK;
        ext = fma(C.cu[d] * b, fx_scaled(fmaf(sk, k, t), emax), ext);
      }
    }
  }
  if (which & (FX_EXT | FX_EXT << 1 | FX_EXT << 2)) atomicAdd(oe, ext);
  int pair = FX_MIXED;
#pragma unroll 1
  for (int q = 0; q < 3; ++q, pair <<= 1) {
    if (!(which & pair)) continue;
    const int si = q < 2 ? 1 : BX, sj = q == 0 ? BX : BX * BX;
    float c = 0.f;
#pragma unroll
    for (int a = 1; a <= H; ++a) {
      float t = 0.f;
#pragma unroll
      for (int b = 1; b <= H; ++b) {
        const float *p = r + a * si, *m = r - a * si;
        t = fmaf((float)X::W1(b), (p[b * sj] - m[b * sj]) - (p[-b * sj] - m[-b * sj]), t);
      }
      c = fmaf((float)X::W1(a), t, c);
    }
    const int o = q == 2 ? 4 : q + 1;
    const double r2 = fx_scaled(c, emax2);
    atomicAdd(o2 + o * vol, C.cubic ? r2 : C.c2[o] * r2);
  }
}

// three limbs of sum_a W1[a] (n_a - n_-a) along stride st, and the largest
// magnitude (high limb) among the n
template <int P>
__device__ __forceinline__ int4 fx_first(const int2* __restrict__ b, int st) {
  long long lo = 0, hi = 0;
  int top = 0, low = 0;
#pragma unroll
  for (int a = 1; a <= FD<P>::H; ++a) {
    const int2 p = b[a * st], m = b[-a * st];
    lo += (long long)FX<P>::W1(a) * (p.x - m.x);
    hi += (long long)FX<P>::W1(a) * (p.y - m.y);
    top = __vimax3_s32(top, p.y, m.y);
    low = __vimin3_s32(low, p.y, m.y);
  }
  hi += lo >> FX_LIMB;
  return make_int4((int)((unsigned int)lo & FX_MASK), (int)((unsigned int)hi & FX_MASK), (int)(hi >> FX_LIMB),
                   max(top, ~low));
}

// the first-derivative weights along stride st of a table of such sums, and
// the largest magnitude among the values they are made of
template <int P>
__device__ __forceinline__ double fx_mixed(const int4* __restrict__ g, int st, int emax, int& mag) {
  long long l0 = 0, l1 = 0;
  int l2 = 0;
  mag = 0;
#pragma unroll
  for (int b = 1; b <= FD<P>::H; ++b) {
    const int4 p = g[b * st], m = g[-b * st];
    l0 += (long long)FX<P>::W1(b) * (p.x - m.x);
    l1 += (long long)FX<P>::W1(b) * (p.y - m.y);
    l2 += FX<P>::W1(b) * (p.z - m.z);
    mag = __vimax3_s32(mag, p.w, m.w);
  }
  l1 += l0 >> FX_LIMB;
  const long long hi = ((long long)(l2 + (int)(l1 >> FX_LIMB)) << FX_LIMB) | (l1 & (long long)FX_MASK);
  return fx_to_double(hi, l0 & (long long)FX_MASK, emax);
}

// The largest magnitude among the values that the upwinded stencil along st reads.
template <int P>
__device__ __noinline__ int fx_upwind_mag(const int2* __restrict__ c, int st) {
  int top = 0, low = 0;
#pragma unroll
  for (int i = 0; i < FD<P>::UPN; ++i) {
    const int v = c[(FD<P>::UPLO + i) * st].y;
    top = max(top, v);
    low = min(low, v);
  }
  return max(top, ~low);
}

// Stencils along the three axes at one point of the box, and the outputs.
// Returns those that fixed point holds too coarsely, where no value that the
// stencil reads is as large as FX_HELD, and << FX_BEYOND those where none is
// even as large as FX_FINE (advection and dissipation leave such axes out, for
// fx_fallback to add). Along an axis the values looked at are those of the
// centred stencils, H on each side. The upwinded stencil does not read the last
// of them on one side: a large value there enters through the dissipation, and
// advection is good to parts in 1e14 of that; where there is little or none
// (weak) its own values are looked at.
template <int P, bool CUBIC, bool D1, bool D2, bool EXT>
__device__ __forceinline__ int fx_point(const int2* __restrict__ c, const int4* const g[3], const FxCoef& C,
                                        const double* beta, bool adv, bool inexact, int emax, int emax1, int emax2,
                                        double* __restrict__ o1, double* __restrict__ o2, double* __restrict__ oe,
                                        int vol) {
  using F = FD<P>;
  using X = FX<P>;
  constexpr int BX = FxSmem<P>::BX;
  const int2 u0 = c[0];
  const int m2x = -2 * u0.x, m2y = -2 * u0.y;
  long long kslo = 0, kshi = 0;
  double ext = 0.0, ko = 0.0;
  int coarse = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int st = d == 0 ? 1 : (d == 1 ? BX : BX * BX);
    int top = 0, low = 0;  // (the point itself is not read by first derivatives)
    int4 f = make_int4(0, 0, 0, 0);  // the sums that mixed derivatives are made of, and their values' magnitude
    if (D2 && d < 2) f = *g[1 + d];
    long long r1l = 0, r1h = 0, r2l = 0, r2h = 0, tl = 0, th = 0, kl = 0, kh = 0;
#pragma unroll
    for (int a = 1; a <= (EXT ? F::R : F::H); ++a) {
      const int2 p = c[a * st], m = c[-a * st];
      const int dx = p.x - m.x, dy = p.y - m.y;
      if (!(D2 && d < 2) && a <= F::H) {
        top = __vimax3_s32(top, p.y, m.y);
        low = __vimin3_s32(low, p.y, m.y);
      }
      if (D1 && !(D2 && d < 2) && a <= F::H) {
        r1l += (long long)X::W1(a) * (dx);
        r1h += (long long)X::W1(a) * (dy);
      }
      if (EXT) {
        tl += (long long)X::WT(a) * (dx);
        th += (long long)X::WT(a) * (dy);
      }
      if (D2 && a <= F::H) {
        const int2 s = fx_pair(p, m);
        r2l += (long long)X::W2(a) * (s.x + m2x);
        r2h += (long long)X::W2(a) * (s.y + m2y);
      }
      if (EXT) {
        kl += (long long)X::WK(a) * (p.x + m.x + m2x);
        kh += (long long)X::WK(a) * (p.y + m.y + m2y);
      }
    }
    const int mag = D2 && d < 2 ? f.w : max(top, ~low);
    bool share = true;
    if (mag < FX_HELD && inexact) {
      const int far = mag < FX_FINE ? 1 | 1 << FX_BEYOND : 1;
      if (D1 || D2) coarse |= far * (FX_AXIS << d);
      if (EXT) coarse |= far * (FX_EXT << d);
      share = mag >= FX_FINE;
    }
    if (EXT && C.weak && inexact && adv) {
      const int um = fx_upwind_mag<P>(c, beta[d] < 0.0 ? -st : st);
      coarse &= ~((1 | 1 << FX_BEYOND) * (FX_EXT << d));
      if (um < FX_HELD) coarse |= (um < FX_FINE ? 1 | 1 << FX_BEYOND : 1) * (FX_EXT << d);
      share = um >= FX_FINE;
    }
    if (D1) {
      if (D2 && d < 2) {
        r1h = ((long long)f.z << FX_LIMB) | (unsigned int)f.y;
        r1l = f.x;
      }
      const double r = fx_to_double(r1h, r1l, emax1);
      o1[d * vol] = CUBIC ? r : C.c1[d] * r;
    }
    if (D2) {
      const double r = fx_to_double(r2h, r2l, emax2);
      o2[sym(d, d) * vol] = CUBIC ? r : C.c2[sym(d, d)] * r;
    }
    if (EXT && share) {
      if (adv) {
        // |beta| times the stencil mirrored by the sign of beta
        const int sk = __double2hiint(beta[d]) < 0 ? -X::SK : X::SK;
        const double U = fx_to_double(th + sk * kh, tl + sk * kl, emax);
        ext = fma(CUBIC ? beta[d] : C.cu[d] * beta[d], U, ext);
      }
      if (CUBIC) {
        kslo += kl;
        kshi += kh;
      } else {
        ko = fma(C.ck[d], fx_to_double(kh, kl, emax), ko);
      }
    }
  }
  if (EXT) *oe = CUBIC ? fma(C.cu[0], ext, C.ck[0] * fx_to_double(kshi, kslo, emax)) : ext + ko;
  if (D2) {
    int mag[3];
    const double xy = fx_mixed<P>(g[0], FX_T, emax2, mag[0]), xz = fx_mixed<P>(g[1], FX_T * FX_T, emax2, mag[1]),
                 yz = fx_mixed<P>(g[2], FX_T * FX_T, emax2, mag[2]);
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (mag[q] < FX_HELD && inexact) coarse |= (mag[q] < FX_FINE ? 1 | 1 << FX_BEYOND : 1) * (FX_MIXED << q);
    o2[1 * vol] = CUBIC ? xy : C.c2[1] * xy;
    o2[2 * vol] = CUBIC ? xz : C.c2[2] * xz;
    o2[4 * vol] = CUBIC ? yz : C.c2[4] * yz;
  }
  return coarse;
}

// The points of a tile's box that its stencils read, in the order they are
// loaded: first the lines through the tile (R points beyond it along one
// axis), then what mixed derivatives add (H beyond it along two). An entry is
// bx | by << 5 | bz << 10 | box index << 16.
template <int P>
struct FxBox {
  static constexpr int H = FD<P>::H, R = FD<P>::R, BX = FX_T + 2 * R;
  static constexpr int LINES = FX_T * FX_T * FX_T + 3 * 2 * R * FX_T * FX_T;
  static constexpr int ALL = LINES + 3 * (2 * H) * (2 * H) * FX_T;
  unsigned int at[ALL];
  constexpr FxBox() : at() {
    int nl = 0, nm = LINES;
    for (int z = 0; z < BX; ++z)
      for (int y = 0; y < BX; ++y)
        for (int x = 0; x < BX; ++x) {
          const int ox = x < R ? R - x : (x >= R + FX_T ? x - (R + FX_T) + 1 : 0);
          const int oy = y < R ? R - y : (y >= R + FX_T ? y - (R + FX_T) + 1 : 0);
          const int oz = z < R ? R - z : (z >= R + FX_T ? z - (R + FX_T) + 1 : 0);
          const int outs = (ox > 0) + (oy > 0) + (oz > 0);
          const unsigned int e = (unsigned int)(x | y << 5 | z << 10 | ((z * BX + y) * BX + x) << 16);
          if (outs <= 1)
            at[nl++] = e;
          else if (outs == 2 && ox <= H && oy <= H && oz <= H)
            at[nm++] = e;
        }
  }
};
template <int P>
__device__ const FxBox<P> g_fx_box{};

// Point of a thread: x and the eight rows of a plane, arranged so that the
// half-warps of an 8-byte shared-memory read take rows y and y + 4, whose
// distance in the box is an odd multiple of 64 bytes (no bank conflicts).
__device__ __forceinline__ void fx_lane(int t, int& x, int& y, int& z) {
  x = t & 7;
  y = ((t >> 3) & 1) * 4 + ((t >> 4) & 1) + ((t >> 5) & 1) * 2;
  z = t >> 6;
}

// Barrier of the threads that work on a tile, the first FX_THREADS of a block.
__device__ __forceinline__ void fx_sync() { asm volatile("bar.sync 1, %0;" ::"n"(FX_THREADS) : "memory"); }

// Does some stencil of a tile of ex x ey x ez points read point (bx, by, bz) of
// its box? (mixed: the variable has mixed derivatives, ext: dissipation, whose
// lines are longer)
template <int P>
__device__ __forceinline__ bool fx_reads(int bx, int by, int bz, int ex, int ey, int ez, bool mixed, bool ext) {
  constexpr int H = FxBox<P>::H, R = FxBox<P>::R;
  const int ox = max(max(R - bx, bx - (R + ex - 1)), 0), oy = max(max(R - by, by - (R + ey - 1)), 0),
            oz = max(max(R - bz, bz - (R + ez - 1)), 0), far = max(ox, max(oy, oz));
  const int axes = (ox > 0) + (oy > 0) + (oz > 0);
  return axes < 2 ? far <= (ext ? R : H) : axes == 2 && mixed && far <= H;
}

// fx_rest of the points of a tile's box (v: its first point, number `first` of
// the `room` points of a variable). Apart from the rest of fx_tile, whose
// registers it would share.
template <int P>
__device__ __noinline__ void fx_rest_box(const double* __restrict__ v, long long first, long long room, long long sy,
                                         long long sz, int ex, int ey, int ez, bool mixed, bool ext, int emax,
                                         float* __restrict__ rest) {
  constexpr int PER = (FxBox<P>::ALL + FX_THREADS - 1) / FX_THREADS;
  const int count = mixed ? FxBox<P>::ALL : FxBox<P>::LINES;
  double raw[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int c = threadIdx.x + q * FX_THREADS;
    raw[q] = 0.0;
    if (c >= count) continue;
    const unsigned int at = __ldg(&g_fx_box<P>.at[c]);
    const int bx = at & 31, by = (at >> 5) & 31, bz = (at >> 10) & 31;
    const long long o = bx + by * sy + bz * sz;
    if (fx_reads<P>(bx, by, bz, ex, ey, ez, mixed, ext) && in_range(first + o, first + o, room)) raw[q] = __ldg(v + o);
  }
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int c = threadIdx.x + q * FX_THREADS;
    if (c < count) rest[__ldg(&g_fx_box<P>.at[c]) >> 16] = fx_rest(raw[q], emax);
  }
}

// All outputs of list entry e on the tile (ti, tj, tk) of the grid L, written
// to the record slot `rec` (nout x vol doubles), by the
// first FX_THREADS threads of the block. box and g: shared memory for the tile
// and its first-derivative tables.
template <int P>
__device__ __forceinline__ void fx_tile(const Layout& L, const FxCoef& C, const FxTiles& T, const DerivList& list,
                                        int e, bool advect_gauge, bool lapse_frozen, bool shift_frozen, bool ko,
                                        const double* __restrict__ u, int ti, int tj, int tk, int2* box, int4* g,
                                        unsigned int (*red)[FX_THREADS / 32], double* __restrict__ rec) {
  using S = FxSmem<P>;
  constexpr int H = S::H, R = S::R, BX = S::BX;

  const int var = list.var[e];
  const bool mixed = list.d2[e] >= 0;
  const int i0 = ti * FX_T, j0 = tj * FX_T, k0 = tk * FX_T;
  const int ex = min(FX_T, L.nx - i0), ey = min(FX_T, L.ny - j0), ez = min(FX_T, L.nz - k0);
  const long long org = L.off0 + i0 + j0 * L.sy + k0 * L.sz;
  const double* __restrict__ v = u + var * L.vs;

  // ---- the box in registers. A ragged tile drops the points that its own
  // stencils do not read (they may lie outside the array, or be ghosts that
  // nothing fills), and so does a variable without dissipation, whose lines
  // are shorter.
  constexpr int PER = (FxBox<P>::ALL + FX_THREADS - 1) / FX_THREADS;
  constexpr int PERL = (FxBox<P>::LINES + FX_THREADS - 1) / FX_THREADS;
  const int count = mixed ? FxBox<P>::ALL : FxBox<P>::LINES;
  const double* __restrict__ v0 = v + (org - R * (1 + L.sy + L.sz));
  const bool d1 = list.d1[e] >= 0, ext = list.ext[e] >= 0;
  const bool full = ex == FX_T && ey == FX_T && ez == FX_T && ext, wide = L.sz >= (1 << 26);
  const int sy = (int)L.sy, sz = (int)L.sz;
  double raw[PER];
  unsigned int at[PER];
  unsigned int mx = 0, any = 0, mn = 0xffffffffu;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    raw[q] = 0.0;
    at[q] = 0xffffffffu;
    if (q >= PERL && !mixed) continue;
    const int c = threadIdx.x + q * FX_THREADS;
    if (c < count) at[q] = __ldg(&g_fx_box<P>.at[c]);
  }
  auto load = [&](auto all) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q >= PERL && !mixed) continue;
      const int bx = at[q] & 31, by = (at[q] >> 5) & 31, bz = (at[q] >> 10) & 31;
      // (a box spans less than 2^31 elements of a variable unless a plane of
      // the array alone has 2^26 points)
      const long long o = wide ? bx + by * L.sy + bz * L.sz : (long long)(bx + by * sy + bz * sz);
      if (decltype(all)::value ? at[q] != 0xffffffffu : fx_reads<P>(bx, by, bz, ex, ey, ez, mixed, ext)) {
        if (in_range(org - R * (1 + L.sy + L.sz) + o, org - R * (1 + L.sy + L.sz) + o, padded_points(L)))
          raw[q] = __ldg(v0 + o);
      }
    }
  };
  if (full)
    load(std::true_type{});
  else
    load(std::false_type{});
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const unsigned int hw = (unsigned int)__double2hiint(raw[q]) & 0x7fffffffu;
    const unsigned int bits = hw | (unsigned int)__double2loint(raw[q]);
    mx = max(mx, hw);
    mn = min(mn, bits ? hw : 0xffffffffu);
    any |= bits;
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  mn = __reduce_min_sync(0xffffffffu, mn);
  any = __reduce_or_sync(0xffffffffu, any);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = mx;
    red[1][threadIdx.x >> 5] = any;
    red[2][threadIdx.x >> 5] = mn;
  }
  fx_sync();
#pragma unroll
  for (int w = 0; w < FX_THREADS / 32; ++w) {
    mx = max(mx, red[0][w]);
    any |= red[1][w];
    mn = min(mn, red[2][w]);
  }
  const bool fallback = mx >= (1900u << 20) || (mx < (160u << 20) && any != 0u);
  const int emax = max((int)(mx >> 20), 160);
  const bool inexact = (int)(mn >> 20) < emax - 6;  // some value loses bits

  const int vol = T.vol;
  const int emax1 = emax + list.s1[e], emax2 = emax + list.s2[e];
  double* const o1 = rec + (long long)(d1 ? list.d1[e] : 0) * vol;
  double* const o2 = rec + (long long)(mixed ? list.d2[e] : 0) * vol;
  double* const oe = rec + (long long)(ext ? list.ext[e] : 0) * vol;
  // does this variable's right-hand side have advection?
  const bool adv = var < V_ALPHA || (advect_gauge && !(var == V_ALPHA ? lapse_frozen : shift_frozen));

  if (!fallback) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q >= PERL && !mixed) continue;
      if (at[q] != 0xffffffffu) box[at[q] >> 16] = fx_from_double(raw[q], emax);
    }
    fx_sync();
    if (mixed) {
      // D_x sums on rows y beyond the tile (for xy) and planes z beyond it
      // (for xz), D_y sums on planes beyond it (for yz); the in-tile D_x
      // serves both tables
      for (int t = threadIdx.x; t < 2 * H * FX_T * FX_T; t += FX_THREADS) {  // xy rows outside
        const int x = t & 7, r = t >> 3, z = r & 7, q = r >> 3;
        const int y = q < H ? q : q + FX_T;  // 0 .. EH-1
        g[(z * S::EH + y) * FX_T + x] = fx_first<P>(box + ((z + R) * BX + (y - H + R)) * BX + x + R, 1);
      }
      for (int t = threadIdx.x; t < S::GN; t += FX_THREADS) {
        int x, y, z;
        fx_lane(t, x, y, z);  // z = 0 .. EH-1
        const int2* b = box + ((z - H + R) * BX + (y + R)) * BX + x + R;
        const int4 fx = fx_first<P>(b, 1);
        g[S::GN + (z * FX_T + y) * FX_T + x] = fx;
        if (z >= H && z < H + FX_T) g[((z - H) * S::EH + (y + H)) * FX_T + x] = fx;
        g[2 * S::GN + (z * FX_T + y) * FX_T + x] = fx_first<P>(b, BX);
      }
      fx_sync();
    }
  }
  // ---- one point per thread
  int x, y, z;
  fx_lane(threadIdx.x, x, y, z);
  const int idx = (z * T.ty + y) * T.tx + x;
  const long long p = org + x + y * L.sy + z * L.sz;
  const bool inside =
      x < ex && y < ey && z < ez && in_range(p - R * L.sz, p + R * L.sz, padded_points(L));
  double beta[3] = {0.0, 0.0, 0.0};
  if (inside && ext && adv)
#pragma unroll
    for (int d = 0; d < 3; ++d) beta[d] = __ldg(u + (V_BETA1 + d) * L.vs + p);
  int coarse = inside && fallback ? FX_ALL | FX_ALL << FX_BEYOND : 0;
  if (inside && !fallback) {
    const int2* c = box + ((z + R) * BX + (y + R)) * BX + x + R;
    const int4* const gt[3] = {g + (z * S::EH + (y + H)) * FX_T + x, g + S::GN + ((z + H) * FX_T + y) * FX_T + x,
                               g + 2 * S::GN + ((z + H) * FX_T + y) * FX_T + x};
    auto point = [&](auto cubic) {
      constexpr bool CB = decltype(cubic)::value;
      double *const p1 = o1 + idx, *const p2 = o2 + idx, *const pe = oe + idx;
      if (mixed && ext)
        return fx_point<P, CB, true, true, true>(c, gt, C, beta, adv, inexact, emax, emax1, emax2, p1, p2, pe, vol);
      if (mixed)
        return fx_point<P, CB, true, true, false>(c, gt, C, beta, adv, inexact, emax, emax1, emax2, p1, p2, pe, vol);
      if (d1 && ext)
        return fx_point<P, CB, true, false, true>(c, gt, C, beta, adv, inexact, emax, emax1, emax2, p1, p2, pe, vol);
      if (d1)
        return fx_point<P, CB, true, false, false>(c, gt, C, beta, adv, inexact, emax, emax1, emax2, p1, p2, pe, vol);
      return fx_point<P, CB, false, false, true>(c, gt, C, beta, adv, inexact, emax, emax1, emax2, p1, p2, pe, vol);
    };
    coarse = C.cubic ? point(std::true_type{}) : point(std::false_type{});
  }
  // ---- where some value lost bits that a point needs, what the integers left
  // out of all of them takes the box's place
  if (!fallback && inexact) {
    const bool some = __any_sync(0xffffffffu, coarse != 0);
    if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = some;
    fx_sync();
    bool tile = false;
#pragma unroll
    for (int w = 0; w < FX_THREADS / 32; ++w) tile |= red[0][w] != 0;
    if (tile) {
      float* rest = (float*)box;
      fx_rest_box<P>(v0, org - R * (1 + L.sy + L.sz), padded_points(L), L.sy, L.sz, ex, ey, ez, mixed, ext, emax, rest);
      fx_sync();
      const int which = coarse & FX_ALL & ~(coarse >> FX_BEYOND);
      if (which)
        fx_refine<P>(rest + ((z + R) * BX + (y + R)) * BX + x + R, C, u + V_BETA1 * L.vs + p, L.vs, adv, which, d1,
                     mixed, emax, emax1, emax2, o1 + idx, o2 + idx, oe + idx, vol);
    }
  }
  if (coarse >> FX_BEYOND)
    fx_fallback<P>(v, p, L.sy, L.sz, C, u + V_BETA1 * L.vs + p, L.vs, adv, ko, coarse >> FX_BEYOND, d1, mixed, ext,
                   list.s1[e] < 0, list.s2[e] < 0, o1 + idx, o2 + idx, oe + idx, vol);
}

// One grid as the FP64 kernels see it: its layout, scales, tiles and buffers.
// Single grids pass one by value; patches keep a device table of them, each
// with the number of its first tile in the flat list of all tiles.
struct FxGrid {
  Layout L;
  FxCoef C;
  FxTiles T;
  long long tile0;
  double* buf[6];  // as PatchDev: 0 y0, 1 and 2 stage buffers, 3 acc, 4 and 5 kept by parents
};

// What a launch works on: a grid passed by value (table null) or the grids
// of a table, tiles tile0, tile0 + 1, ... of the flat list, slot by slot.
struct FxWork {
  FxGrid one;
  const FxGrid* table;
  const long long* tile0s;  // first tile of every grid of the table
  int ngrids;
  long long tile0;          // tile of slot 0
  double* rec;
  long long slot;           // doubles of one slot
};

// grid and tile coordinates of a slot
__device__ __forceinline__ const FxGrid& fx_locate(const FxWork& Wk, long long t, int& ti, int& tj, int& tk) {
  const FxGrid* G = &Wk.one;
  if (Wk.table) {
    int lo = 0, hi = Wk.ngrids - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(Wk.tile0s + mid) <= t) lo = mid; else hi = mid - 1;
    }
    G = Wk.table + lo;
  }
  const unsigned int q = (unsigned int)(t - G->tile0);
  const unsigned int r = q / (unsigned int)G->T.ntx;
  ti = (int)(q - r * G->T.ntx);
  tk = (int)(r / (unsigned int)G->T.nty);
  tj = (int)(r - tk * (unsigned int)G->T.nty);
  return *G;
}

struct DerivArgs {
  FxWork W;
  DerivList list;
  int in;  // buffer the stencils read
  bool advect_gauge, lapse_frozen, shift_frozen;
  bool ko;  // a stage (its dissipation may be 0); a right-hand side alone has none
};

// What a thread does with the right-hand side of its point.
struct StageOut {
  int mode;                // 0: RK stage, 1: right-hand side to out
  Gauge gz;
  RK rk;
  int in, out;             // buffers of the stage input and of the result
  double* rhs;             // mode 1: where the right-hand side goes
};

struct AlgebraArgs {
  FxWork W;
  StageOut S;
};

// One block per slot (blockIdx.x) and list entry (blockIdx.y).
template <int P>
__global__ void __launch_bounds__(FX_THREADS, 2) k_derivs(const __grid_constant__ DerivArgs A) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  int4* g = (int4*)fx_smem;
  int ti, tj, tk;
  const int e = blockIdx.y;
  const FxGrid& G = fx_locate(A.W, A.W.tile0 + blockIdx.x, ti, tj, tk);
  const double* u = G.buf[A.in];
  __shared__ unsigned int red[3][FX_THREADS / 32];
  fx_tile<P>(G.L, G.C, G.T, A.list, e, A.advect_gauge, A.lapse_frozen, A.shift_frozen, A.ko, u,
             ti, tj, tk, (int2*)(g + 3 * FxSmem<P>::GN), g, red,
             A.W.rec + (long long)blockIdx.x * A.W.slot);
}

}  // namespace bssn
