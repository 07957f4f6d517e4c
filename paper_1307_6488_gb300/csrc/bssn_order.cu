// Instantiates the kernels and launchers for one finite-difference order,
// selected at compile time with -DBSSN_ORDER=4 or -DBSSN_ORDER=8.
#include "bssn_fixed.cuh"
#include "bssn_kernels.cuh"
#include "bssn_weyl.cuh"
#include "bssn_launch.h"
#include "bssn_bounds.cuh"

#ifndef BSSN_ORDER
#error "compile with -DBSSN_ORDER=4 or -DBSSN_ORDER=8"
#endif

namespace bssn {

static inline unsigned int blocks_for(long long n, int threads) { return (unsigned int)((n + threads - 1) / threads); }

template <>
cudaError_t launch_diffs<BSSN_ORDER>(const Layout& L, const double* u, double* dX, double* dY, cudaStream_t s) {
  constexpr int H = FD<BSSN_ORDER>::H;
  const long long n = (long long)L.nx * (L.ny + 2 * H) * (L.nz + 2 * H);
  k_diffs<BSSN_ORDER, double><<<blocks_for(n, 256), 256, 0, s>>>(L, u, dX, dY);
  return cudaGetLastError();
}

static std::atomic<unsigned long long> g_derivs_smem{0};  // devices whose limit is raised

template <>
cudaError_t derivs_init<BSSN_ORDER>() {
  return allow_smem(k_derivs<BSSN_ORDER>, FxSmem<BSSN_ORDER>::bytes, g_derivs_smem);
}

template <>
cudaError_t launch_derivs<BSSN_ORDER>(const DerivArgs& A, long long nslots, cudaStream_t s) {
  constexpr size_t bytes = FxSmem<BSSN_ORDER>::bytes;
  const cudaError_t e = derivs_init<BSSN_ORDER>();
  if (e != cudaSuccess) return e;
  k_derivs<BSSN_ORDER><<<dim3((unsigned int)nslots, (unsigned int)A.list.n), FX_THREADS, bytes, s>>>(A);
  return cudaGetLastError();
}

template <>
cudaError_t launch_ko<BSSN_ORDER>(const Layout& L, const bssn_grid_t& G, double eps, bssn_precision_t prec,
                                  const double* u, double* rhs, cudaStream_t s) {
  if (prec == BSSN_FP64)
    k_ko<BSSN_ORDER, double><<<blocks_for(L.npts, 256), 256, 0, s>>>(L, make_coef<BSSN_ORDER, double>(G, eps), u, rhs);
  else
    k_ko<BSSN_ORDER, float><<<blocks_for(L.npts, 256), 256, 0, s>>>(L, make_coef<BSSN_ORDER, float>(G, eps), u, rhs);
  return cudaGetLastError();
}

template <>
cudaError_t launch_constraints<BSSN_ORDER>(const Layout& L, const Coef<double>& C, const double* u,
                                           const double* dX, const double* dY, double* ham, double* mom,
                                           double* gcon, double* part, unsigned int* flag, bool ham_only,
                                           cudaStream_t s) {
  if (ham_only)
    k_constraints<BSSN_ORDER, true><<<(unsigned int)con_blocks(L), CON_THREADS, 0, s>>>(L, C, u, dX, dY, ham,
                                                                                        nullptr, nullptr, part, flag);
  else
    k_constraints<BSSN_ORDER, false><<<(unsigned int)con_blocks(L), CON_THREADS, 0, s>>>(L, C, u, dX, dY, ham, mom,
                                                                                         gcon, part, flag);
  return cudaGetLastError();
}

template <>
cudaError_t launch_psi4<BSSN_ORDER>(const Layout& L, const Coef<double>& C, const double* u, const double* dX,
                                    const double* dY, const double origin[3], const double h[3], double* psi_re,
                                    double* psi_im, double* inv_re, double* inv_im, double* E, double* B,
                                    unsigned int* flag, cudaStream_t s) {
  k_psi4<BSSN_ORDER><<<blocks_for(L.npts, 128), 128, 0, s>>>(L, C, u, dX, dY, origin[0], origin[1], origin[2], h[0],
                                                             h[1], h[2], psi_re, psi_im, inv_re, inv_im, E, B,
                                                             flag);
  return cudaGetLastError();
}


template <>
cudaError_t bounds_take_order<BSSN_ORDER>(unsigned long long* out) {
  return bounds_take_local(out);
}

}  // namespace bssn
