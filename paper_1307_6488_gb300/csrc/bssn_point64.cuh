// Pointwise algebra of the FP64 forms: the right-hand side of the BSSN system
// (the equations at the head of bssn_point.cuh), the Hamiltonian constraint
// and the conformal Ricci tensor, written for as few FP64 instructions as
// possible (the kernels that use it are bound by the FP64 pipe; the stage's
// executes ~800 per point with its update, 1176 with the algebra the FP32 form
// uses: at 128^3, 8th order, 8.33 -> 7.74 ms per stage when made, derivatives
// included). The momentum and Gamma constraints have a form of their own
// (momentum64).
//
//  * Half the metric's first derivatives come from the record, so Christoffel
//    symbols of the first kind are sums of them, most of them a single one.
//  * With P_i^km = gt^ml Gt^k_li the quadratic terms of the Ricci tensor are
//      2 Gt^k_l(i Gt_j)k^l + Gt^k_im Gt_kj^m
//        = P_i^km d_m gt_jk + P_j^km Gt_i,km,
//    because Gt_j,km + Gt_k,jm = d_m gt_jk; likewise
//    Gd^k (Gt_i,jk + Gt_j,ik) = Gd^k d_k gt_ij.
//  * Only the trace-free part of -D_i D_j alpha + alpha R_ij is needed, so
//    its terms proportional to gt_ij are never formed; the trace of D_i D_j
//    alpha is written out.
//  * Terms linear in one tensor are gathered first (Au^ij times one vector,
//    gt^ij times one vector, Gt^k_ij times one vector).
#pragma once
#include "bssn_common.cuh"
#include "bssn_point.cuh"

namespace bssn {

// One point's derivatives, as the record scales them: first derivatives 1/a
// times and second derivatives 1/a2 = 1/a^2 times their value, where a, a2 and
// b = a2 / a are what the functions below take (FxCoef).
struct Point64 {
  double u[NV];
  double dW[3], dK[3], da[3];
  double hg[3][6];    // 1/2 d_d gt_s
  double hG[3][3];    // hG[d][i] = 1/2 d_d Gt^i
  double db[3][3];    // db[d][i] = d_d beta^i
  double ddW[6], dda[6];
  double ddb[3][6];   // d_s beta^i
  double hgg[6][6];   // hgg[s][t] = 1/2 d_t gt_s
};

// Christoffel symbols in the first derivatives' units, Ricci in the second's.
struct Conformal64 {
  double gu[6], gu2[6];  // gt^ij; with off-diagonal entries doubled
  double GU[3][6];       // Gt^k_ij
  double Gd[3];          // gt^ij Gt^k_ij
  double R[6];           // conformal Ricci tensor
};

// ia = 1 / a brings d Gt^k to the second derivatives' units
__device__ __forceinline__ void conformal64(const Point64& P, double ia, Conformal64& C) {
  const double* g = P.u + V_GT11;
  {
    const double c0 = g[3] * g[5] - g[4] * g[4];
    const double c1 = g[2] * g[4] - g[1] * g[5];
    const double c2 = g[1] * g[4] - g[2] * g[3];
    const double c3 = g[0] * g[5] - g[2] * g[2];
    const double c4 = g[1] * g[2] - g[0] * g[4];
    const double c5 = g[0] * g[3] - g[1] * g[1];
    const double idet = 1.0 / (g[0] * c0 + g[1] * c1 + g[2] * c2);
    C.gu[0] = c0 * idet; C.gu[1] = c1 * idet; C.gu[2] = c2 * idet;
    C.gu[3] = c3 * idet; C.gu[4] = c4 * idet; C.gu[5] = c5 * idet;
#pragma unroll
    for (int s = 0; s < 6; ++s) C.gu2[s] = (s == 1 || s == 2 || s == 4) ? C.gu[s] + C.gu[s] : C.gu[s];
  }
  // Gt_k,ij = 1/2 (d_i gt_kj + d_j gt_ki - d_k gt_ij)
  double GL[3][6];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const int i = sym_i(s), j = sym_j(s);
      if (k == i)
        GL[k][s] = P.hg[j][sym(i, i)];
      else if (k == j)
        GL[k][s] = P.hg[i][sym(j, j)];
      else if (i == j)
        GL[k][s] = fma(2.0, P.hg[i][sym(k, i)], -P.hg[k][s]);
      else
        GL[k][s] = P.hg[i][sym(k, j)] + (P.hg[j][sym(k, i)] - P.hg[k][s]);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int s = 0; s < 6; ++s)
      C.GU[k][s] = C.gu[sym(k, 0)] * GL[0][s] + C.gu[sym(k, 1)] * GL[1][s] + C.gu[sym(k, 2)] * GL[2][s];
    double t = C.gu2[0] * C.GU[k][0];
#pragma unroll
    for (int s = 1; s < 6; ++s) t = fma(C.gu2[s], C.GU[k][s], t);
    C.Gd[k] = t;
  }
  // terms linear in second derivatives, d Gt^k and Gd^k
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int i = sym_i(s), j = sym_j(s);
    double r = C.Gd[0] * P.hg[0][s];
#pragma unroll
    for (int k = 1; k < 3; ++k) r = fma(C.Gd[k], P.hg[k][s], r);
#pragma unroll
    for (int t = 0; t < 6; ++t) r = fma(-C.gu2[t], P.hgg[s][t], r);
    double l = g[sym(i, 0)] * P.hG[j][0] + g[sym(i, 1)] * P.hG[j][1] + g[sym(i, 2)] * P.hG[j][2];
    if (i == j) {
      r = fma(ia + ia, l, r);
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) l = fma(g[sym(j, k)], P.hG[i][k], l);
      r = fma(ia, l, r);
    }
    C.R[s] = r;
  }
  // quadratic terms, index i of P_i^km at a time: P_i^km d_m gt_jk for every
  // pair s = (i, j) whose first index is i, P_i^km Gt_a,km for every pair
  // (a, i) whose second index is i
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double Pm[3][3];  // Pm[k][m] = P_i^km
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int m = 0; m < 3; ++m)
        Pm[k][m] = C.gu[sym(m, 0)] * C.GU[k][sym(0, i)] + C.gu[sym(m, 1)] * C.GU[k][sym(1, i)] +
                   C.gu[sym(m, 2)] * C.GU[k][sym(2, i)];
#pragma unroll
    for (int j = i; j < 3; ++j) {
      double t = Pm[0][0] * P.hg[0][sym(j, 0)];
#pragma unroll
      for (int km = 1; km < 9; ++km) t = fma(Pm[km / 3][km % 3], P.hg[km % 3][sym(j, km / 3)], t);
      C.R[sym(i, j)] = fma(2.0, t, C.R[sym(i, j)]);
    }
    const double p1 = Pm[0][1] + Pm[1][0], p2 = Pm[0][2] + Pm[2][0], p4 = Pm[1][2] + Pm[2][1];
#pragma unroll
    for (int a = 0; a <= i; ++a) {
      double t = C.R[sym(a, i)];
      t = fma(Pm[0][0], GL[a][0], t);
      t = fma(p1, GL[a][1], t);
      t = fma(p2, GL[a][2], t);
      t = fma(Pm[1][1], GL[a][3], t);
      t = fma(p4, GL[a][4], t);
      C.R[sym(a, i)] = fma(Pm[2][2], GL[a][5], t);
    }
  }
}

// Right-hand side of the 24 variables added to rhs (which holds advection and
// dissipation on entry). gz.lapse / gz.shift as in bssn_point.cuh.
__device__ __forceinline__ void rhs_point64(const Point64& P, const Gauge& gz, double a, double a2, double ia,
                                            double b, double rhs[NV]) {
  Conformal64 C;
  conformal64(P, ia, C);
  const double* u = P.u;
  const double* g = u + V_GT11;
  const double* A = u + V_AT11;
  const double W = u[V_W], K = u[V_TRK], al = u[V_ALPHA], al2 = al + al;
  const double iW = 1.0 / W, W2 = a2 * (W * W);  // W2 only ever multiplies second derivatives
  const double third = 1.0 / 3.0, twothirds = 2.0 / 3.0;
  double db[3][3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int i = 0; i < 3; ++i) db[d][i] = a * P.db[d][i];
  const double div = db[0][0] + db[1][1] + db[2][2], d23 = twothirds * div;

  double dWs[3];  // d_i W / W
#pragma unroll
  for (int i = 0; i < 3; ++i) dWs[i] = P.dW[i] * iW;

  // X_ij = -D_i D_j alpha + alpha R_ij without its terms in gt_ij
  double X[6], trX;
  {
    const double aw = al * iW;
    double v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = fma(aw, P.dW[k], -P.da[k]);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const int i = sym_i(s), j = sym_j(s);
      double x = fma(al, C.R[s], fma(aw, P.ddW[s], -P.dda[s]));
#pragma unroll
      for (int k = 0; k < 3; ++k) x = fma(-C.GU[k][s], v[k], x);
      if (i == j)
        x = fma(-2.0 * dWs[i], P.da[i], x);
      else
        x = fma(-dWs[i], P.da[j], fma(-dWs[j], P.da[i], x));
      X[s] = x;
    }
    trX = C.gu2[0] * X[0];
#pragma unroll
    for (int s = 1; s < 6; ++s) trX = fma(C.gu2[s], X[s], trX);
  }
  // gt^ij D_i D_j alpha = gt^ij d_i d_j alpha - Gd^k d_k alpha - gt^ij d_i W d_j alpha / W
  double lap = C.gu2[0] * P.dda[0];
#pragma unroll
  for (int s = 1; s < 6; ++s) lap = fma(C.gu2[s], P.dda[s], lap);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    lap = fma(-C.Gd[k], P.da[k], lap);
    const double wu = C.gu[sym(k, 0)] * dWs[0] + C.gu[sym(k, 1)] * dWs[1] + C.gu[sym(k, 2)] * dWs[2];
    lap = fma(-wu, P.da[k], lap);
  }

  // At^i_j, At^ij (off-diagonal entries doubled in Au2)
  double Am[3][3], Au[6], Au2[6];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Am[i][j] = C.gu[sym(i, 0)] * A[sym(0, j)] + C.gu[sym(i, 1)] * A[sym(1, j)] + C.gu[sym(i, 2)] * A[sym(2, j)];
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int i = sym_i(s), j = sym_j(s);
    Au[s] = Am[i][0] * C.gu[sym(0, j)] + Am[i][1] * C.gu[sym(1, j)] + Am[i][2] * C.gu[sym(2, j)];
    Au2[s] = i == j ? Au[s] : Au[s] + Au[s];
  }
  double AA = A[0] * Au2[0];
#pragma unroll
  for (int s = 1; s < 6; ++s) AA = fma(A[s], Au2[s], AA);

  rhs[V_W] = fma(third * W, al * K - div, rhs[V_W]);
  rhs[V_TRK] = fma(-W2, lap, fma(al, fma(third * K, K, AA), rhs[V_TRK]));
  const double cX = third * W2 * trX, cA = fma(al, K, -d23);
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int i = sym_i(s), j = sym_j(s);
    double rg = fma(-al2, A[s], fma(-d23, g[s], rhs[V_GT11 + s]));
    double ra = fma(W2, X[s], fma(-cX, g[s], fma(cA, A[s], rhs[V_AT11 + s])));
    const double aa = A[sym(i, 0)] * Am[0][j] + A[sym(i, 1)] * Am[1][j] + A[sym(i, 2)] * Am[2][j];
    ra = fma(-al2, aa, ra);
    double lg = g[sym(i, 0)] * db[j][0] + g[sym(i, 1)] * db[j][1] + g[sym(i, 2)] * db[j][2];
    double la = A[sym(i, 0)] * db[j][0] + A[sym(i, 1)] * db[j][1] + A[sym(i, 2)] * db[j][2];
    if (i == j) {
      rg = fma(2.0, lg, rg);
      ra = fma(2.0, la, ra);
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        lg = fma(g[sym(j, k)], db[i][k], lg);
        la = fma(A[sym(j, k)], db[i][k], la);
      }
      rg += lg;
      ra += la;
    }
    rhs[V_GT11 + s] = rg;
    rhs[V_AT11 + s] = ra;
  }

  double q[3], w[3];  // what At^ij and gt^ij are contracted with
  const double a6 = -6.0 * al, a43 = (-4.0 / 3.0) * al, b3 = third * b;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    q[j] = fma(a6, dWs[j], -2.0 * P.da[j]);
    w[j] = fma(a43, P.dK[j], b3 * (P.ddb[0][sym(j, 0)] + P.ddb[1][sym(j, 1)] + P.ddb[2][sym(j, 2)]));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    // everything in units of one first derivative; the second derivatives of
    // beta, the largest terms where beta is rough, are added last
    double t6 = Au2[0] * C.GU[i][0];
    double lap = C.gu2[0] * P.ddb[i][0];
#pragma unroll
    for (int s = 1; s < 6; ++s) {
      t6 = fma(Au2[s], C.GU[i][s], t6);
      lap = fma(C.gu2[s], P.ddb[i][s], lap);
    }
    double r = fma(d23, C.Gd[i], al2 * t6);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      r = fma(Au[sym(i, j)], q[j], r);
      r = fma(-C.Gd[j], db[j][i], r);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) r = fma(C.gu[sym(i, j)], w[j], r);
    r = fma(b, lap, r);
    rhs[V_GAM1 + i] = fma(a, r, rhs[V_GAM1 + i]);
    if (gz.shift == 0) {
      rhs[V_BETA1 + i] = fma(gz.shift_coeff, u[V_B1 + i], rhs[V_BETA1 + i]);
      rhs[V_B1 + i] = fma(a, r, fma(-gz.eta, u[V_B1 + i], rhs[V_B1 + i]));
    }
  }
  if (gz.lapse == 0)
    rhs[V_ALPHA] = fma(-al2, K, rhs[V_ALPHA]);
  else if (gz.lapse == 1)
    rhs[V_ALPHA] = fma(-al * al, K, rhs[V_ALPHA]);
}

// Hamiltonian constraint at a point.
__device__ __forceinline__ double hamiltonian64(const Point64& P, double a2, double ia) {
  Conformal64 C;
  conformal64(P, ia, C);
  const double* A = P.u + V_AT11;
  const double W = P.u[V_W], K = P.u[V_TRK];
  // gt^ij R_ij: the conformal part, and 4 gt^ij DtDt_ij W / W - 6 gt^ij d_i W d_j W / W^2
  double tr = C.gu2[0] * C.R[0], tw = C.gu2[0] * P.ddW[0], ww = 0.0;
#pragma unroll
  for (int s = 1; s < 6; ++s) {
    tr = fma(C.gu2[s], C.R[s], tr);
    tw = fma(C.gu2[s], P.ddW[s], tw);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    tw = fma(-C.Gd[k], P.dW[k], tw);
    ww = fma(C.gu[sym(k, 0)] * P.dW[0] + C.gu[sym(k, 1)] * P.dW[1] + C.gu[sym(k, 2)] * P.dW[2], P.dW[k], ww);
  }
  double Am[3][3], AA = 0.0;  // At^i_j
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Am[i][j] = C.gu[sym(i, 0)] * A[sym(0, j)] + C.gu[sym(i, 1)] * A[sym(1, j)] + C.gu[sym(i, 2)] * A[sym(2, j)];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) AA = fma(Am[i][j], Am[j][i], AA);
  // W^2 R = W^2 tr + 4 W tw - 6 ww
  return fma(a2, fma(W, fma(W, tr, 4.0 * tw), -6.0 * ww), fma((2.0 / 3.0) * K, K, -AA));
}

// First derivative along a stride: sum_a c_a (u_a - u_-a).
template <int H>
__device__ __forceinline__ double d1_direct(const double* __restrict__ v, long long s, const double* c) {
  double r = c[1] * (__ldg(v + s) - __ldg(v - s));
#pragma unroll
  for (int a = 2; a <= H; ++a) r = fma(c[a], __ldg(v + a * s) - __ldg(v - a * s), r);
  return r;
}

// What the momentum and Gamma constraints and the magnetic part of the Weyl
// tensor are made of, from the state itself: first derivatives by stencils in
// double precision and the Christoffel symbols.
//
// On data that satisfies the constraints these are what is left of terms that
// cancel: on a gauge wave (A = 0.05, noise 1e-10) terms of order 1 leave 1e-8 to
// 1e-10, and parts in 1e-9 to 1e-8 of the result are the rounding of whatever
// form is evaluated. This form is the one that their values have always had, so
// they stay the same to the last bit; from the derivative record, rounded once
// and gathered differently, they were as close to a quadruple-precision
// evaluation but up to 9e-9 of their norm apart from these. All constraints at
// 128^3, 8th order: 12.0 ms with every stencil in double precision, 6.4 with
// these alone, 4.0 with none.
struct First64 {
  double u[V_ALPHA];  // the variables up to Gt^i
  double dW[3], dK[3], dg[3][6], dAt[3][6];
  double gu[6], gu2[6];  // gt^ij; with off-diagonal entries doubled
  double GU[3][6], Gd[3];  // Gt^k_ij, gt^ij Gt^k_ij
};

// c1: the first-derivative weights over the spacing
template <int H>
__device__ __forceinline__ void first64(const double* __restrict__ up, long long vs, const long long st[3],
                                        const double (*c1)[5], First64& F) {
#pragma unroll
  for (int v = 0; v < V_ALPHA; ++v) F.u[v] = __ldg(up + v * vs);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    F.dW[d] = d1_direct<H>(up + V_W * vs, st[d], c1[d]);
    F.dK[d] = d1_direct<H>(up + V_TRK * vs, st[d], c1[d]);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      F.dg[d][s] = d1_direct<H>(up + (V_GT11 + s) * vs, st[d], c1[d]);
      F.dAt[d][s] = d1_direct<H>(up + (V_AT11 + s) * vs, st[d], c1[d]);
    }
  }
  double GL[3][6];  // Gt_k,ij
  inverse_metric<double>(F.u + V_GT11, F.gu);
#pragma unroll
  for (int s = 0; s < 6; ++s) F.gu2[s] = (s == 1 || s == 2 || s == 4) ? F.gu[s] + F.gu[s] : F.gu[s];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const int i = sym_i(s), j = sym_j(s);
      GL[k][s] = 0.5 * (F.dg[i][sym(k, j)] + F.dg[j][sym(k, i)] - F.dg[k][s]);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int s = 0; s < 6; ++s)
      F.GU[k][s] = F.gu[sym(k, 0)] * GL[0][s] + F.gu[sym(k, 1)] * GL[1][s] + F.gu[sym(k, 2)] * GL[2][s];
    double t = F.gu2[0] * F.GU[k][0];
#pragma unroll
    for (int s = 1; s < 6; ++s) t += F.gu2[s] * F.GU[k][s];
    F.Gd[k] = t;
  }
}

// Momentum (out[0..2]) and Gamma (out[3..5]) constraints.
__device__ __forceinline__ void momentum64(const First64& F, double out[6]) {
  const double iW = 1.0 / F.u[V_W];
  const double* A = F.u + V_AT11;
  double Am[3][3];  // At^i_j
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      Am[i][j] = F.gu[sym(i, 0)] * A[sym(0, j)] + F.gu[sym(i, 1)] * A[sym(1, j)] + F.gu[sym(i, 2)] * A[sym(2, j)];
  // M_i = gt^jk (d_k At_ij - Gt^l_ki At_lj - Gt^l_kj At_il) - 3/W At^j_i d_j W - 2/3 d_i K
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double div = 0.0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {  // twice the summand, symmetrised over (j, k)
      const int j = sym_i(s), k = sym_j(s);
      double t = F.dAt[k][sym(i, j)] + F.dAt[j][sym(i, k)];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        t -= F.GU[l][sym(k, i)] * A[sym(l, j)] + F.GU[l][sym(k, j)] * A[sym(i, l)];
        t -= F.GU[l][sym(j, i)] * A[sym(l, k)] + F.GU[l][sym(j, k)] * A[sym(i, l)];
      }
      div += F.gu2[s] * t;
    }
    const double aw = Am[0][i] * F.dW[0] + Am[1][i] * F.dW[1] + Am[2][i] * F.dW[2];
    out[i] = 0.5 * div - 3.0 * iW * aw - (2.0 / 3.0) * F.dK[i];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) out[3 + i] = F.u[V_GAM1 + i] - F.Gd[i];
}

}  // namespace bssn
