// The FP64 stage of single grids, patches and refined levels: derivatives on
// the integer pipes (k_derivs, bssn_fixed.cuh), then the pointwise algebra
// and the stage update on the FP64 pipe, tile by tile through a record that
// holds as many tiles as the caller's scratch takes.
#include <algorithm>

#include "bssn_bounds.cuh"
#include "bssn_fixed.cuh"
#include "bssn_launch.h"
#include "bssn_point.cuh"

namespace bssn {

// Threads of a block and resident blocks per SM. The kernel is bound by the
// FP64 pipe (~1100 instructions per point at 1.68 per clock and SM), which a
// few warps keep busy; small blocks spread a small grid over all SMs.
#ifndef ALG_THREADS
#define ALG_THREADS 64
#endif
#ifndef ALG_MIN_BLOCKS
#define ALG_MIN_BLOCKS 4
#endif

// One thread per point of a slot: the pointwise right-hand side from the
// record of k_derivs, plus its advection + dissipation sums, and the stage
// update.
__global__ void __launch_bounds__(ALG_THREADS, ALG_MIN_BLOCKS) k_algebra(const __grid_constant__ AlgebraArgs A,
                                                                       int blocks_per_slot) {
  const unsigned int slot = blockIdx.x / (unsigned int)blocks_per_slot;
  const int idx = (int)(blockIdx.x - slot * blocks_per_slot) * ALG_THREADS + threadIdx.x;
  int ti, tj, tk;
  const FxGrid& G = fx_locate(A.W, A.W.tile0 + slot, ti, tj, tk);
  const Layout& L = G.L;
  const int vol = G.T.vol;
  if (idx >= vol) return;
  const int x = idx % G.T.tx, yz = idx / G.T.tx;
  const int i = ti * FX_T + x, j = tj * FX_T + yz % G.T.ty, k = tk * FX_T + yz / G.T.ty;
  if (i >= L.nx || j >= L.ny || k >= L.nz) return;
  const long long p = L.off0 + i + j * L.sy + k * L.sz;
  if (!in_range(p, p, padded_points(L))) return;
  const long long vs = L.vs;
  const double* __restrict__ rec = A.W.rec + (long long)slot * A.W.slot + idx;
  const double* __restrict__ ys = G.buf[A.S.in] + p;
  PointIn<double> Q;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    Q.u[v] = __ldg(ys + v * vs);
    Q.adv[v] = 0.0;  // added below, with the dissipation
  }
  auto r = [&](int o) { return __ldg(rec + o * vol); };
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Q.dW[d] = r(d);
    Q.da[d] = r(9 * 7 + d);
    Q.dK[d] = r(REC_K + d);
#pragma unroll
    for (int s = 0; s < 6; ++s) Q.dg[d][s] = r(9 * (1 + s) + d);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Q.db[d][c] = r(9 * (8 + c) + d);
      Q.dGam[d][c] = r(REC_GAM + 3 * c + d);
    }
  }
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    Q.ddW[s] = r(3 + s);
    Q.dda[s] = r(9 * 7 + 3 + s);
#pragma unroll
    for (int c = 0; c < 3; ++c) Q.ddb[c][s] = r(9 * (8 + c) + 3 + s);
#pragma unroll
    for (int c = 0; c < 6; ++c) Q.ddg[c][s] = r(9 * (1 + c) + 3 + s);
  }
  double rhs[NV];
  rhs_point<double>(Q, A.S.gz, 1.0 / Q.u[V_W], rhs);
#pragma unroll
  for (int v = 0; v < NV; ++v) rhs[v] += r(REC_EXT + v);
  if (A.S.mode == 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v) A.S.rhs[v * vs + p] = rhs[v];
    return;
  }
  const RK& rk = A.S.rk;
  const double* y0 = G.buf[0] + p;  // may be the output: read before it is written
  double* acc = G.buf[3] + p;
  double* out = G.buf[A.S.out] + p;
  if (rk.method == 3) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const long long o = v * vs;
      out[o] = fma(rk.cdt, rhs[v], fma(rk.a1, Q.u[v], rk.a0 * y0[o]));
    }
    return;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const long long o = v * vs;
    double yn;
    if (rk.stage == 0) {
      acc[o] = rk.bdt * rhs[v];
      yn = fma(rk.cdt, rhs[v], y0[o]);
    } else if (rk.stage < 3) {
      acc[o] = fma(rk.bdt, rhs[v], acc[o]);
      yn = fma(rk.cdt, rhs[v], y0[o]);
    } else {
      yn = y0[o] + fma(rk.bdt, rhs[v], acc[o]);
    }
    out[o] = yn;
  }
}

cudaError_t launch_stage64(int order, const FxWork& work, int vol, long long ntiles, long long slots,
                           const Gauge& gz, const StageOut& out, cudaStream_t s) {
  if (slots < 1) return cudaErrorInvalidValue;
  const long long chunks = (ntiles + slots - 1) / slots, per = (ntiles + chunks - 1) / chunks;
  DerivArgs D{work, rhs_list(), out.in, gz.advect_gauge != 0, gz.lapse == 2, gz.shift == 1};
  AlgebraArgs A{work, out};
  const int bps = (vol + ALG_THREADS - 1) / ALG_THREADS;
  for (long long t = 0; t < ntiles; t += per) {
    const long long n = std::min(per, ntiles - t);
    D.W.tile0 = A.W.tile0 = work.tile0 + t;
    const cudaError_t e = order == 4 ? launch_derivs<4>(D, n, s) : launch_derivs<8>(D, n, s);
    if (e != cudaSuccess) return e;
    k_algebra<<<(unsigned int)(n * bps), ALG_THREADS, 0, s>>>(A, bps);
    const cudaError_t e2 = cudaGetLastError();
    if (e2 != cudaSuccess) return e2;
  }
  return cudaSuccess;
}

cudaError_t bounds_take_stage64(unsigned long long* out) { return bounds_take_local(out); }

}  // namespace bssn
