// Batched RK4 stepping of many uneven grid patches (the single-GPU analogue
// of the block-structured AMR/multi-block grids the paper plans for, Sec. 4
// and Sec. 1.1; tile selection prior art, Sec. 2.6).
//
// A plan holds, for every patch, three stage buffers (and in the FP32-RHS
// form two single-precision copies and derivative tables), device tables that
// describe the patches, in FP64 the derivative record, and one CUDA graph per
// step size. One RK4 step of all patches is one graph launch: four times
// (static ghost fill, stage), then a final ghost fill. A stage is the single
// grids' kernels over the tiles of all patches: k_derivs and k_algebra in
// FP64 (bssn_stage64.cu), tables and k_stage32t_batch in the FP32-RHS form (the
// first stage also converts the state). No device-side waiting between blocks, no
// sums across threads, and a deterministic result; the per-point arithmetic is
// the single grids'.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <tuple>
#include <vector>

#include "../../include/bssn.h"
#include "bssn_launch.h"
#include "bssn_patch.cuh"

using namespace bssn;

struct bssn_plan {
  int np = 0;
  int order = 4;
  bssn_precision_t prec = BSSN_FP64;
  bssn_params_t params{};
  Gauge gz{};
  std::vector<PatchDev> host;
  PatchDev* dev = nullptr;
  long long* d_gh0 = nullptr;
  long long ntiles = 0, nghost = 0, points = 0;
  std::vector<void*> allocations;
  int shape = 0;  // tile shape index bssn_plan_info reports
  int grid_other = 0;
  // FP64 form: the patches as the stage kernels see them, and their record
  FxTable fx;
  double* rec = nullptr;
  // FP32-RHS form: the tiled kernels of bssn_stage32.cuh over a second table,
  // ordered by spacing so that each spacing's patches are one range,
  // and numbered by that order; two tables that differ in the single-precision
  // copy of the state, the second absent where there was no memory for it
  std::vector<Patch32> host32;  // of the first
  Patch32* dev32[2] = {nullptr, nullptr};
  long long* d_tile32 = nullptr;
  long long* d_pad32 = nullptr;
  long long* d_ext32 = nullptr;
  long long ntiles32 = 0, npad32 = 0, next32 = 0;
  struct Level {
    int p0, np;
    long long tbase, ntiles;
    Coef32 C;
  };
  std::vector<Level> levels;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  double graph_dt = NAN;
  cudaStream_t cap = nullptr;
};

namespace {

cudaError_t plan_alloc(bssn_plan* pl, size_t bytes, void** out) {
  cudaError_t e = cudaMalloc(out, bytes);
  if (e == cudaSuccess) pl->allocations.push_back(*out);
  return e;
}

void plan_free(bssn_plan* pl) {
  if (pl->exec) cudaGraphExecDestroy(pl->exec);
  if (pl->graph) cudaGraphDestroy(pl->graph);
  if (pl->cap) cudaStreamDestroy(pl->cap);
  for (void* p : pl->allocations) cudaFree(p);
  pl->allocations.clear();
}

// Static ghosts of buffer `which` of every patch (and of the single-precision
// copies of the table p32, nullable).
cudaError_t fill_all(bssn_plan* pl, int which, const Patch32* p32, cudaStream_t s) {
  kb_fill<<<dim3((unsigned int)pl->grid_other, NV / 4), 256, 0, s>>>(pl->dev, p32, pl->d_gh0, pl->np, pl->nghost,
                                                                     which);
  return cudaGetLastError();
}

// The second single-precision copies and their table, one allocation, made
// last: a plan that finds no memory for them converts the input of every
// stage instead. Entry i of the table is the patch with slot32 == i.
cudaError_t second_copies(bssn_plan* pl, const bssn_block_t* blocks) {
  const size_t table = sizeof(Patch32) * pl->np;
  auto copy_bytes = [](const Patch32& Q) { return ((size_t)NV * Q.L32.vs * sizeof(float) + 255) & ~(size_t)255; };
  size_t bytes = 0;
  for (const Patch32& Q : pl->host32) bytes += copy_bytes(Q);
  void* p = nullptr;
  cudaError_t e = plan_alloc(pl, bytes + table, &p);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return cudaSuccess;
  }
  if (e != cudaSuccess) return e;
  std::vector<Patch32> t = pl->host32;
  char* f = (char*)p;
  for (int b = 0; b < pl->np; ++b) {
    Patch32& Q = t[pl->host[b].slot32];
    const Patch32 A = Q;
    const bool ok =
        pl->order == 4
            ? make_patch32<4>(&Q, blocks[b].grid, pl->params.ko_eps, pl->host[b].buf, (float*)f, A.tab)
            : make_patch32<8>(&Q, blocks[b].grid, pl->params.ko_eps, pl->host[b].buf, (float*)f, A.tab);
    if (!ok) return cudaErrorInvalidValue;
    f += copy_bytes(A);
  }
  pl->dev32[1] = (Patch32*)f;
  return cudaMemcpy(f, t.data(), table, cudaMemcpyHostToDevice);
}

// One FP32-RHS stage of all patches with the tiled kernels: single-precision
// copy of the stage input (where `convert`; otherwise the stage before and the
// ghost fill wrote it), D_x / D_y tables, then one stage launch per spacing,
// which also writes the copies of the table `next` (nullable).
cudaError_t stage32_all(bssn_plan* pl, const RK& rk, int in, int out, const Patch32* cur, const Patch32* next,
                        bool convert, cudaStream_t s) {
  const int g = pl->grid_other;
  cudaError_t e = convert ? launch_to_f32t_batch(cur, pl->d_pad32, pl->np, pl->npad32, in, g, s) : cudaSuccess;
  if (e == cudaSuccess)
    e = pl->order == 4 ? launch_d1tab32_batch<4>(cur, pl->d_ext32, pl->np, pl->next32, g, s)
                       : launch_d1tab32_batch<8>(cur, pl->d_ext32, pl->np, pl->next32, g, s);
  for (const auto& lv : pl->levels) {
    if (e != cudaSuccess) break;
    e = pl->order == 4 ? launch_stage32_batch<4>(cur, next, pl->d_tile32, lv.p0, lv.np, lv.tbase, lv.ntiles, lv.C,
                                                 pl->gz, rk, in, out, s)
                       : launch_stage32_batch<8>(cur, next, pl->d_tile32, lv.p0, lv.np, lv.tbase, lv.ntiles, lv.C,
                                                 pl->gz, rk, in, out, s);
  }
  return e;
}

// The launch sequence of one RK4 step (captured into the graph).
cudaError_t enqueue_step(bssn_plan* pl, double dt, cudaStream_t s) {
  const int ins[4] = {0, 1, 2, 1};
  const int outs[4] = {1, 2, 1, 0};
  cudaError_t e = cudaSuccess;
  for (int st = 0; st < 4 && e == cudaSuccess; ++st) {
    // the first stage converts the state; the others find the copy that the
    // stage before wrote (interior) and this fill completes (ghosts), the two
    // copies in turn: the same values without three conversion passes (23.9 ->
    // 22.5 ms per step of 96 uneven 4th-order patches)
    const bool two = pl->dev32[1], convert = st == 0 || !two;
    const Patch32* cur = pl->dev32[two ? st & 1 : 0];
    e = fill_all(pl, ins[st], convert ? nullptr : cur, s);
    if (e != cudaSuccess) break;
    const RK rk = make_rk(st, dt);
    e = pl->prec == BSSN_FP32_RHS
            ? stage32_all(pl, rk, ins[st], outs[st], cur, two && st < 3 ? pl->dev32[1 - (st & 1)] : nullptr, convert, s)
            : fx_stage(pl->order, pl->fx, pl->rec, pl->gz, rk, ins[st], outs[st], s);
  }
  if (e == cudaSuccess) e = fill_all(pl, 0, nullptr, s);
  return e;
}

}  // namespace

namespace bssn {
cudaError_t bounds_take_batch(unsigned long long* out) { return bounds_take_local(out); }
}  // namespace bssn

extern "C" {

bssn_status_t bssn_plan_create(bssn_plan_t** out, const bssn_block_t* blocks, int nblocks,
                               const bssn_params_t* params, bssn_precision_t prec, int autotune) {
  if (!out || !blocks || nblocks < 1 || nblocks > (1 << 20) || !params) return BSSN_ERR_INVALID_ARG;
  if (prec != BSSN_FP64 && prec != BSSN_FP32_RHS) return BSSN_ERR_INVALID_ARG;
  *out = nullptr;
  for (int b = 0; b < nblocks; ++b) {
    const bssn_block_t& B = blocks[b];
    if (bssn_work_bytes(&B.grid, params, prec) == 0) return BSSN_ERR_INVALID_ARG;
    if (!B.state || !B.ghost_src || ((uintptr_t)B.state & 15) || ((uintptr_t)B.ghost_src & 15))
      return BSSN_ERR_INVALID_ARG;
    if (B.state == B.ghost_src) return BSSN_ERR_INVALID_ARG;
  }
  bssn_plan* pl = new (std::nothrow) bssn_plan;
  if (!pl) return BSSN_ERR_NOMEM;
  pl->np = nblocks;
  pl->order = params->fd_order;
  pl->prec = prec;
  pl->params = *params;
  pl->gz = make_gauge(*params);
  pl->host.resize(nblocks);
  cudaError_t e = cudaSuccess;
  const int H = pl->order / 2;
  std::vector<long long> gh0(nblocks);
  for (int b = 0; b < nblocks && e == cudaSuccess; ++b) {
    const bssn_block_t& B = blocks[b];
    PatchDev& D = pl->host[b];
    std::memset((void*)&D, 0, sizeof(D));
    D.L = make_layout(B.grid);
    D.buf[0] = B.state;
    D.ghost = B.ghost_src;
    const size_t n = (size_t)NV * B.grid.var_stride;
    void* p = nullptr;
    e = plan_alloc(pl, 3 * n * sizeof(double), &p);
    if (e != cudaSuccess) break;
    D.buf[1] = (double*)p;
    D.buf[2] = D.buf[1] + n;
    D.buf[3] = D.buf[2] + n;
    // stage buffers start as a copy of the state so their ghosts are defined
    e = cudaMemcpy(D.buf[1], B.state, n * sizeof(double), cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(D.buf[2], B.state, n * sizeof(double), cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess) e = cudaMemset(D.buf[3], 0, n * sizeof(double));
    if (e != cudaSuccess) break;
    D.gh0 = gh0[b] = pl->nghost;
    pl->nghost += ghost_points(D.L);
    pl->points += D.L.npts;
  }
  void* p = nullptr;
  // FP32-RHS: per patch a single-precision copy and tables in Layout32, and
  // the tiled kernels' table, sorted by spacing (one stage launch each)
  if (e == cudaSuccess && prec == BSSN_FP32_RHS) {
    std::vector<int> ord(nblocks);
    for (int b = 0; b < nblocks; ++b) ord[b] = b;
    std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) {
      const bssn_grid_t &A = blocks[a].grid, &Bg = blocks[b].grid;
      return std::make_tuple(A.dx, A.dy, A.dz) < std::make_tuple(Bg.dx, Bg.dy, Bg.dz);
    });
    pl->host32.resize(nblocks);
    std::vector<long long> t0(nblocks), q0(nblocks), x0(nblocks);
    long long nt = 0, nq = 0, nx = 0;
    for (int i = 0; i < nblocks && e == cudaSuccess; ++i) {
      const int b = ord[i];
      const bssn_grid_t& G = blocks[b].grid;
      const Layout32 L32 = make_layout32(G);
      e = plan_alloc(pl, (size_t)(NV + 2 * NM) * L32.vs * sizeof(float), &p);
      if (e != cudaSuccess) break;
      float* f32 = (float*)p;
      float* tab = f32 + (size_t)NV * L32.vs;
      Patch32& Q = pl->host32[i];
      std::memset((void*)&Q, 0, sizeof(Q));
      const bool ok = pl->order == 4 ? make_patch32<4>(&Q, G, params->ko_eps, pl->host[b].buf, f32, tab)
                                     : make_patch32<8>(&Q, G, params->ko_eps, pl->host[b].buf, f32, tab);
      if (!ok) {
        e = cudaErrorInvalidValue;
        break;
      }
      pl->host[b].slot32 = i;
      Q.tile0 = t0[i] = nt;
      nt += (long long)Q.ntx * Q.nty * ((G.nz + 3) / 4);
      Q.pad0 = q0[i] = nq;
      nq += (G.nx + 2LL * G.ghost) * (G.ny + 2LL * G.ghost) * (G.nz + 2LL * G.ghost);
      Q.ext0 = x0[i] = nx;
      nx += (long long)G.nx * (G.ny + 2 * H) * (G.nz + 2 * H);
      if (i == 0 || G.dx != blocks[ord[i - 1]].grid.dx || G.dy != blocks[ord[i - 1]].grid.dy ||
          G.dz != blocks[ord[i - 1]].grid.dz)
        pl->levels.push_back({i, 0, Q.tile0, 0, Q.C});
      pl->levels.back().np += 1;
      pl->levels.back().ntiles = nt - pl->levels.back().tbase;
    }
    pl->ntiles32 = nt;
    pl->npad32 = nq;
    pl->next32 = nx;
    if (e == cudaSuccess) e = plan_alloc(pl, sizeof(Patch32) * nblocks, &p);
    if (e == cudaSuccess) {
      pl->dev32[0] = (Patch32*)p;
      e = cudaMemcpy(p, pl->host32.data(), sizeof(Patch32) * nblocks, cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) e = plan_alloc(pl, 3 * sizeof(long long) * nblocks, &p);
    if (e == cudaSuccess) {
      pl->d_tile32 = (long long*)p;
      pl->d_pad32 = pl->d_tile32 + nblocks;
      pl->d_ext32 = pl->d_pad32 + nblocks;
    }
    if (e == cudaSuccess) e = cudaMemcpy(pl->d_tile32, t0.data(), sizeof(long long) * nblocks, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(pl->d_pad32, q0.data(), sizeof(long long) * nblocks, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(pl->d_ext32, x0.data(), sizeof(long long) * nblocks, cudaMemcpyHostToDevice);
    pl->shape = 6;  // the tiled kernel's 8 x 4 x 4
    pl->ntiles = nt;
    if (e == cudaSuccess) e = pl->order == 4 ? stage32_batch_init<4>() : stage32_batch_init<8>();
  }
  if (e == cudaSuccess && prec == BSSN_FP64) {
    std::vector<FxGrid> grids;
    for (int b = 0; b < nblocks; ++b) grids.push_back(fx_grid(blocks[b].grid, pl->order, params->ko_eps, pl->host[b].buf));
    e = fx_upload(grids, &pl->fx, [&](size_t n, void** q) { return plan_alloc(pl, n, q); });
    pl->ntiles = pl->fx.ntiles;
    if (e == cudaSuccess) e = plan_alloc(pl, pl->fx.record_doubles() * sizeof(double), &p);
    if (e == cudaSuccess) pl->rec = (double*)p;
    if (e == cudaSuccess) e = pl->order == 4 ? derivs_init<4>() : derivs_init<8>();
  }
  if (e == cudaSuccess) e = plan_alloc(pl, sizeof(PatchDev) * nblocks, &p);
  if (e == cudaSuccess) {
    pl->dev = (PatchDev*)p;
    e = cudaMemcpy(pl->dev, pl->host.data(), sizeof(PatchDev) * nblocks, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = plan_alloc(pl, sizeof(long long) * nblocks, &p);
  if (e == cudaSuccess) {
    pl->d_gh0 = (long long*)p;
    e = cudaMemcpy(pl->d_gh0, gh0.data(), sizeof(long long) * nblocks, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&pl->cap, cudaStreamNonBlocking);
  int dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  pl->grid_other = 8 * std::max(1, sms);
  if (e == cudaSuccess && prec == BSSN_FP32_RHS) e = second_copies(pl, blocks);
  if (e != cudaSuccess) {
    plan_free(pl);
    delete pl;
    return e == cudaErrorMemoryAllocation ? BSSN_ERR_NOMEM : BSSN_ERR_CUDA;
  }
  *out = pl;
  return BSSN_OK;
}

bssn_status_t bssn_batch_step(bssn_plan_t* pl, double dt, void* stream) {
  if (!pl || !std::isfinite(dt)) return BSSN_ERR_INVALID_ARG;
  cudaError_t e = cudaSuccess;
  if (!pl->exec || pl->graph_dt != dt) {
    if (pl->exec) { cudaGraphExecDestroy(pl->exec); pl->exec = nullptr; }
    if (pl->graph) { cudaGraphDestroy(pl->graph); pl->graph = nullptr; }
    e = cudaStreamBeginCapture(pl->cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      cudaError_t e2 = enqueue_step(pl, dt, pl->cap);
      e = cudaStreamEndCapture(pl->cap, &pl->graph);
      if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&pl->exec, pl->graph, 0);
    if (e != cudaSuccess) return BSSN_ERR_CUDA;
    pl->graph_dt = dt;
  }
  e = cudaGraphLaunch(pl->exec, (cudaStream_t)stream);
  return e == cudaSuccess ? BSSN_OK : BSSN_ERR_CUDA;
}

bssn_status_t bssn_plan_info(const bssn_plan_t* pl, long long* points, long long* tiles, int* shapes) {
  if (!pl) return BSSN_ERR_INVALID_ARG;
  if (points) *points = pl->points;
  if (tiles) *tiles = pl->ntiles;
  if (shapes)
    for (int b = 0; b < pl->np; ++b) shapes[b] = pl->shape;
  return BSSN_OK;
}

bssn_status_t bssn_plan_destroy(bssn_plan_t* pl) {
  if (!pl) return BSSN_ERR_INVALID_ARG;
  plan_free(pl);
  delete pl;
  return BSSN_OK;
}

}  // extern "C"
