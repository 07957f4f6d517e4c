// Instantiates the kernels and launchers for one finite-difference order,
// selected at compile time with -DBSSN_ORDER=4 or -DBSSN_ORDER=8.
#include "bssn_fixed.cuh"
#include "bssn_ko.cuh"
#include "bssn_stage64.cuh"
#include "bssn_launch.h"
#include "bssn_bounds.cuh"

#ifndef BSSN_ORDER
#error "compile with -DBSSN_ORDER=4 or -DBSSN_ORDER=8"
#endif

namespace bssn {

static inline unsigned int blocks_for(long long n, int threads) { return (unsigned int)((n + threads - 1) / threads); }

static std::atomic<unsigned long long> g_derivs_smem{0}, g_overlap_smem{0};  // devices whose limit is raised

template <>
cudaError_t derivs_init<BSSN_ORDER>() {
  const cudaError_t e = allow_smem(k_derivs<BSSN_ORDER>, FxSmem<BSSN_ORDER>::bytes, g_derivs_smem);
  return e == cudaSuccess ? allow_smem(k_overlap<BSSN_ORDER>, FxSmem<BSSN_ORDER>::bytes, g_overlap_smem) : e;
}

template <>
cudaError_t launch_overlap<BSSN_ORDER>(const OverlapArgs& A, int sms, cudaStream_t s) {
  const cudaError_t e = derivs_init<BSSN_ORDER>();
  if (e != cudaSuccess) return e;
  k_overlap<BSSN_ORDER><<<sms, OVERLAP_THREADS<BSSN_ORDER>, FxSmem<BSSN_ORDER>::bytes, s>>>(A);
  return cudaGetLastError();
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
cudaError_t bounds_take_order<BSSN_ORDER>(unsigned long long* out) {
  return bounds_take_local(out);
}

}  // namespace bssn
