// Patches of a block-structured grid as the batched and the refined-
// hierarchy steppers see them: the device description of one patch, the
// ghost-fill kernel that walks a flat list of all patches' points (grid-
// stride: no device-side waiting, no atomics), and the FP64 stage over a
// table of patches. Included by
// bssn_batch.cu and bssn_amr.cu; everything has internal linkage (an unnamed
// namespace at file scope, like the rest of those files).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "bssn_bounds.cuh"
#include "bssn_cvt.cuh"
#include "bssn_launch.h"

namespace {
using namespace bssn;

// Device description of one patch.
struct PatchDev {
  Layout L;
  long long gh0;            // first point of this patch in the flat ghost-point list
  int slot32;               // FP32-RHS plans: the patch's place in the Patch32 tables
  double* buf[6];           // 0: state (y0, result), 1: ya, 2: yb, 3: acc; parents in a
                            // refined hierarchy also 4: third stage input, 5: y0 kept
  const double* ghost;      // t = 0 state: source of the static ghosts
};

__device__ __forceinline__ int find_patch(const long long* __restrict__ start, int n, long long t) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(start + mid) <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// --- persistent kernels over all patches -------------------------------------------------

// Static ghosts: copy every ghost point of `which` buffer from the t = 0 state,
// the variables 4 blockIdx.y ... of it (as k_fill_ghosts), and, where P32 is
// given, into that table's single-precision copies.
__global__ void __launch_bounds__(256) kb_fill(const PatchDev* __restrict__ P, const Patch32* __restrict__ P32,
                                              const long long* __restrict__ gh0, int np, long long total, int which) {
  constexpr int FILL_VARS = 4;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int b = find_patch(gh0, np, t);
    const PatchDev& D = P[b];
    const Layout& L = D.L;
    int i, j, k;
    ghost_point(L, t - D.gh0, i, j, k);
    const long long p = L.off0 + i + j * L.sy + k * L.sz;
    if (!in_range(p, p, padded_points(L))) continue;
    double* u = D.buf[which] + p + blockIdx.y * FILL_VARS * L.vs;
    const double* src = D.ghost + p + blockIdx.y * FILL_VARS * L.vs;
    double x[FILL_VARS];
#pragma unroll
    for (int v = 0; v < FILL_VARS; ++v) x[v] = __ldg(src + v * L.vs);
#pragma unroll
    for (int v = 0; v < FILL_VARS; ++v) u[v * L.vs] = x[v];
    if (P32) {
      const Patch32& Q = P32[D.slot32];
      const long long q = idx32(Q.L32, i, j, k);
      if (!in_range(q, q, padded_points32(Q.L32))) continue;
      float* f = Q.f32 + q + blockIdx.y * FILL_VARS * Q.L32.vs;
#pragma unroll
      for (int v = 0; v < FILL_VARS; ++v) f[v * Q.L32.vs] = f64_to_f32_rn(x[v]);
    }
  }
}

// The FP64 stage's view of a list of patches: the device table of FxGrid
// entries and the first tile of each, and a record that all stages share.
struct FxTable {
  FxGrid* dev = nullptr;
  long long* tile0s = nullptr;
  int n = 0;
  int vol = 1;              // points of the largest tile
  long long ntiles = 0;
  long long slots = 0;      // tiles of its record, and the record's size
  size_t record_doubles() const { return (size_t)slots * REC_RHS * vol; }
};

// Slots of the shared record: at most this many tiles are between the two
// kernels of a stage at a time (1.1 GB where tiles have 512 points).
constexpr long long FX_MAX_SLOTS = 2048;

FxGrid fx_grid(const bssn_grid_t& G, int order, double eps, double* const buf[6]) {
  FxGrid F{};
  F.L = make_layout(G);
  F.C = order == 4 ? make_fx<4>(G, eps) : make_fx<8>(G, eps);
  F.T = fx_tiles(G.nx, G.ny, G.nz);
  for (int k = 0; k < 6; ++k) F.buf[k] = buf[k];
  return F;
}

// Number the tiles of `grids` and upload the table (alloc: cudaMalloc that
// the owner frees).
template <typename Alloc>
cudaError_t fx_upload(std::vector<FxGrid>& grids, FxTable* T, Alloc alloc) {
  std::vector<long long> t0(grids.size());
  T->n = (int)grids.size();
  T->ntiles = 0;
  for (size_t b = 0; b < grids.size(); ++b) {
    grids[b].tile0 = t0[b] = T->ntiles;
    T->ntiles += (long long)grids[b].T.ntx * grids[b].T.nty * grids[b].T.ntz;
    T->vol = std::max(T->vol, grids[b].T.vol);
  }
  T->slots = std::min(FX_MAX_SLOTS, stage64_slots(T->ntiles));
  void* p = nullptr;
  cudaError_t e = alloc(sizeof(FxGrid) * grids.size(), &p);
  T->dev = (FxGrid*)p;
  if (e == cudaSuccess) e = alloc(sizeof(long long) * grids.size(), &p);
  T->tile0s = (long long*)p;
  if (e == cudaSuccess) e = cudaMemcpy(T->dev, grids.data(), sizeof(FxGrid) * grids.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(T->tile0s, t0.data(), sizeof(long long) * t0.size(), cudaMemcpyHostToDevice);
  return e;
}

// One FP64 stage of every patch of the table, buffer `in` to buffer `out`,
// through a record of at least T.record_doubles().
cudaError_t fx_stage(int order, const FxTable& T, double* rec, const Gauge& gz, const RK& rk, int in, int out,
                     cudaStream_t s) {
  FxWork W{};
  W.table = T.dev;
  W.tile0s = T.tile0s;
  W.ngrids = T.n;
  W.rec = rec;
  W.slot = (long long)REC_RHS * T.vol;
  return launch_stage64(order, W, T.vol, T.ntiles, T.slots, gz, StageOut{0, gz, rk, in, out, nullptr}, s);
}

}  // namespace
