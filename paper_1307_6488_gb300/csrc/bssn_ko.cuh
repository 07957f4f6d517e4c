// Kreiss-Oliger dissipation alone (bssn_ko_dissipation), templated on the
// finite-difference order P and the arithmetic type R.
#pragma once
#include "bssn_common.cuh"

namespace bssn {

__device__ __forceinline__ double fmaR(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmaR(float a, float b, float c) { return fmaf(a, b, c); }

template <int P, typename R>
__global__ void __launch_bounds__(256) k_ko(Layout L, Coef<R> C, const double* __restrict__ u, double* rhs) {
  using F = FD<P>;
  const long long lin = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (lin >= L.npts) return;
  const int i = (int)(lin % L.nx);
  const long long row = lin / L.nx;
  const int j = (int)(row % L.ny), k = (int)(row / L.ny);
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

}  // namespace bssn
