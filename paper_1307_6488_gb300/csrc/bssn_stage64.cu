// The FP64 stage of single grids, patches and refined levels, the constraints
// and the Weyl scalars: derivatives on the integer pipes (k_derivs,
// bssn_fixed.cuh), then the pointwise algebra on the FP64 pipe, tile by tile
// through a record that holds as many tiles as the caller's scratch takes (the
// momentum and Gamma constraints and the magnetic Weyl part make their own,
// first64).
#include <algorithm>

#include "bssn_bounds.cuh"
#include "bssn_fixed.cuh"
#include "bssn_launch.h"
#include "bssn_stage64.cuh"
#include "bssn_weyl.cuh"

namespace bssn {

// Threads of a block and resident blocks per SM. The kernel is bound by the
// FP64 pipe (~800 instructions per point at 1.68 per clock and SM), which a
// few warps keep busy; small blocks spread a small grid over all SMs.
#ifndef ALG_THREADS
#define ALG_THREADS 64
#endif
#ifndef ALG_MIN_BLOCKS
#define ALG_MIN_BLOCKS 4
#endif

__global__ void __launch_bounds__(ALG_THREADS, ALG_MIN_BLOCKS) k_algebra(const __grid_constant__ AlgebraArgs A,
                                                                       int blocks_per_slot) {
  const unsigned int slot = blockIdx.x / (unsigned int)blocks_per_slot;
  algebra_point<PART_ALL>(A.W, A.S, slot, (int)(blockIdx.x - slot * blocks_per_slot) * ALG_THREADS + threadIdx.x);
}

// The same for few points: At_ij and the other variables by different warps.
// A warp's FP64 instruction holds its scheduler's FP64 unit for 64 clocks
// whatever the other schedulers do, so where not every scheduler has a warp
// the time is that of one warp's instructions, and two halves (with their
// shared part done twice) take about half of it.
__global__ void __launch_bounds__(32) k_algebra_split(const __grid_constant__ AlgebraArgs A, int groups) {
  const unsigned int q = blockIdx.x >> 1, slot = q / (unsigned int)groups;
  const int idx = (int)(q - slot * groups) * 32 + threadIdx.x;
  if (blockIdx.x & 1)
    algebra_point<PART_REST>(A.W, A.S, slot, idx);
  else
    algebra_point<PART_AT>(A.W, A.S, slot, idx);
}

// Algebra of n slots, split where that is shorter: where whole warps would
// leave schedulers without one (one RK4 step of 24^3 points, 27 tiles, 298 ->
// 271 us; of 32 x 24 x 24, 36 tiles, 328 -> 332, so not there), and where the
// schedulers' last whole warp is the only one of most of them (40 x 32 x 32, 80
// tiles, 738 -> 658 us; 36^3 901 -> 831; with fewer than two warps each it does
// not pay, 32 x 32 x 24 425 -> 433). A half takes about 0.55 of a warp's time.
static cudaError_t launch_algebra(const AlgebraArgs& A, long long n, int vol, int schedulers, cudaStream_t s) {
  const int groups = (vol + 31) / 32;
  const long long warps = n * groups;
  auto rounds = [&](long long w) { return (w + schedulers - 1) / schedulers; };
  if (2 * warps <= schedulers + schedulers / 2 ||
      (warps > 2 * schedulers && 0.55 * rounds(2 * warps) < (double)rounds(warps))) {
    k_algebra_split<<<(unsigned int)(2 * n * groups), 32, 0, s>>>(A, groups);
  } else {
    const int bps = (vol + ALG_THREADS - 1) / ALG_THREADS;
    k_algebra<<<(unsigned int)(n * bps), ALG_THREADS, 0, s>>>(A, bps);
  }
  return cudaGetLastError();
}

// What the Hamiltonian constraint and the conformal Ricci tensor take, at one point.
__device__ __forceinline__ void load_ham(const double* __restrict__ rec, int vol, const double* __restrict__ u,
                                         long long vs, Point64& Q) {
  auto r = [&](int o) { return __ldg(rec + o * vol); };
#pragma unroll
  for (int v = 0; v < NV; ++v) Q.u[v] = __ldg(u + v * vs);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Q.dW[d] = r(d);
#pragma unroll
    for (int s = 0; s < 6; ++s) Q.hg[d][s] = r(9 * (1 + s) + d);
#pragma unroll
    for (int c = 0; c < 3; ++c) Q.hG[d][c] = r(REC_C_GAM + 3 * c + d);
  }
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    Q.ddW[s] = r(3 + s);
#pragma unroll
    for (int c = 0; c < 6; ++c) Q.hgg[c][s] = r(9 * (1 + c) + 3 + s);
  }
}

struct ConArgs {
  FxWork W;
  double *ham, *mom, *gcon, *part;
  unsigned int* flag;
  double c1[3][5];  // first-derivative weights over the spacing
};

// Constraints of the points of `nblocks` blocks of CON_THREADS points
// (blocks_per_slot to a slot), grid-stride. Per-block partial results, 7 sums
// of squares and 7 maxima, are added to part[blockIdx.x * 14 + q] (written by
// the first chunk), so that one small array serves any number of tiles in a
// fixed order. H = 0: the Hamiltonian constraint alone (the momentum and
// Gamma slots stay 0); its values are the same bits as in the full evaluation.
// H = p/2: the momentum and Gamma constraints too, from the state itself
// (first64). Bound by the FP64 pipe (128 registers and 4 blocks an SM, as
// the algebra).
template <int H>
__global__ void __launch_bounds__(CON_THREADS, 4) k_constraints(const __grid_constant__ ConArgs A, unsigned int nblocks,
                                                               int blocks_per_slot, bool first) {
  double sum[7], top[7];
#pragma unroll
  for (int q = 0; q < 7; ++q) sum[q] = top[q] = 0.0;
  bool bad = false;
  for (unsigned int b = blockIdx.x; b < nblocks; b += gridDim.x) {
    const unsigned int slot = b / (unsigned int)blocks_per_slot;
    const int idx = (int)(b - slot * blocks_per_slot) * CON_THREADS + threadIdx.x;
    int ti, tj, tk;
    const FxGrid& G = fx_locate(A.W, A.W.tile0 + slot, ti, tj, tk);
    TilePoint pt;
    if (!tile_point(G, ti, tj, tk, idx, pt)) continue;
    const long long p = pt.p, vs = G.L.vs;
    const double* __restrict__ u = G.buf[1] + p;
    double c[7];
    if constexpr (H > 0) {
      if (!in_range(p - H * G.L.sz, p + H * G.L.sz, padded_points(G.L))) continue;
      const long long st[3] = {1, G.L.sy, G.L.sz};
      First64 F;
      first64<H>(u, vs, st, A.c1, F);
      momentum64(F, c + 1);
      if (A.mom)
#pragma unroll
        for (int a = 0; a < 3; ++a) A.mom[a * vs + p] = c[1 + a];
      if (A.gcon)
#pragma unroll
        for (int a = 0; a < 3; ++a) A.gcon[a * vs + p] = c[4 + a];
#pragma unroll
      for (int q = 1; q < 7; ++q) {
        bad |= !isfinite(c[q]);
        sum[q] += c[q] * c[q];
        top[q] = fmax(top[q], fabs(c[q]));  // a NaN is left out here and reported by the flag
      }
    }
    Point64 Q;
    load_ham(A.W.rec + (long long)slot * A.W.slot + idx, G.T.vol, u, vs, Q);
    c[0] = hamiltonian64(Q, G.C.a2, G.C.ia);
    if (A.ham) A.ham[p] = c[0];
    bad |= !isfinite(c[0]);
    sum[0] += c[0] * c[0];
    top[0] = fmax(top[0], fabs(c[0]));
    bad |= !(Q.u[V_W] > 0.0);  // the conformal factor must stay positive
  }
  if (bad) atomicOr(A.flag, 1u);
  __shared__ double red[CON_THREADS / 32][14];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    double s = sum[q], m = top[q];
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
    double* out = A.part + (long long)blockIdx.x * 14 + q;
    double r = first ? 0.0 : *out;
    for (int w = 0; w < CON_THREADS / 32; ++w) r = (q < 7) ? r + red[w][q] : fmax(r, red[w][q]);
    *out = r;
  }
}

struct WeylArgs {
  FxWork W;
  double o[3], h[3];
  double *psi_re, *psi_im, *inv_re, *inv_im, *E, *B;
  unsigned int* flag;
  double c1[3][5];  // first-derivative weights over the spacing
};

// Weyl scalars, one point per thread; outputs in the state's padded layout
// (E and B as 6 arrays var_stride apart), each nullable. The conformal Ricci
// tensor comes from the record, the rest from the state (first64, H = p/2).
// FP64-pipe bound.
template <int H>
__global__ void __launch_bounds__(CON_THREADS, 4) k_psi4(const __grid_constant__ WeylArgs A, int blocks_per_slot) {
  const unsigned int slot = blockIdx.x / (unsigned int)blocks_per_slot;
  const int idx = (int)(blockIdx.x - slot * blocks_per_slot) * CON_THREADS + threadIdx.x;
  int ti, tj, tk;
  const FxGrid& G = fx_locate(A.W, A.W.tile0 + slot, ti, tj, tk);
  TilePoint pt;
  if (!tile_point(G, ti, tj, tk, idx, pt)) return;
  const long long p = pt.p, vs = G.L.vs;
  if (!in_range(p - H * G.L.sz, p + H * G.L.sz, padded_points(G.L))) return;
  const double* __restrict__ u = G.buf[1] + p;
  double ddW[6], R[6];
  {
    Point64 Q;
    load_ham(A.W.rec + (long long)slot * A.W.slot + idx, G.T.vol, u, vs, Q);
    Conformal64 C;
    conformal64(Q, G.C.ia, C);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      ddW[s] = Q.ddW[s] * G.C.a2;
      R[s] = C.R[s] * G.C.a2;
    }
  }
  First64 F;
  const long long st[3] = {1, G.L.sy, G.L.sz};
  first64<H>(u, vs, st, A.c1, F);
  const double xyz[3] = {A.o[0] + pt.i * A.h[0], A.o[1] + pt.j * A.h[1], A.o[2] + pt.k * A.h[2]};
  WeylOut O;
  weyl_point(F, ddW, R, xyz, O);
  const bool bad = !isfinite(O.psi_re) || !isfinite(O.psi_im) || !isfinite(O.inv_re) || !isfinite(O.inv_im);
  if (A.psi_re) A.psi_re[p] = O.psi_re;
  if (A.psi_im) A.psi_im[p] = O.psi_im;
  if (A.inv_re) A.inv_re[p] = O.inv_re;
  if (A.inv_im) A.inv_im[p] = O.inv_im;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    if (A.E) A.E[s * vs + p] = O.E[s];
    if (A.B) A.B[s * vs + p] = O.B[s];
  }
  if (bad) atomicOr(A.flag, 1u);
}

// Runs derivatives and `use` (called with the slots of the chunk and whether
// it is the first) over the grid's tiles, as many at a time as the record holds.
template <typename F>
static cudaError_t through_record(int order, const FxWork& work, const DerivList& list, size_t rec_doubles,
                                  cudaStream_t s, F use) {
  const FxTiles& T = work.one.T;
  DerivArgs D{work, list, 1, false, false, false, false};
  D.W.slot = (long long)list.nout * T.vol;
  const long long ntiles = (long long)T.ntx * T.nty * T.ntz, slots = (long long)(rec_doubles / (size_t)D.W.slot);
  if (slots < 1) return cudaErrorInvalidValue;
  const long long chunks = (ntiles + slots - 1) / slots, per = (ntiles + chunks - 1) / chunks;
  for (long long t = 0; t < ntiles; t += per) {
    const long long n = std::min(per, ntiles - t);
    D.W.tile0 = t;
    cudaError_t e = order == 4 ? launch_derivs<4>(D, n, s) : launch_derivs<8>(D, n, s);
    if (e != cudaSuccess) return e;
    use(D.W, n, t == 0);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

static void first_weights(int order, const double h[3], double c1[3][5]) {
  for (int d = 0; d < 3; ++d)
    for (int a = 1; a <= order / 2; ++a) c1[d][a] = (order == 4 ? FD<4>::W1[a] : FD<8>::W1[a]) / h[d];
}

cudaError_t launch_constraints(int order, FxWork work, const double h[3], size_t rec_doubles, double* ham, double* mom,
                               double* gcon, double* part, long long max_parts, int* nparts, unsigned int* flag,
                               bool ham_only, cudaStream_t s) {
  ConArgs A{work, ham, mom, gcon, part, flag, {}};
  first_weights(order, h, A.c1);
  const int bps = (work.one.T.vol + CON_THREADS - 1) / CON_THREADS;
  *nparts = 0;
  return through_record(order, work, ham_list(), rec_doubles, s, [&](const FxWork& W, long long n, bool first) {
    A.W = W;
    // as many blocks as are resident (4 on each of 152 SMs): each takes the
    // points of several tiles, and the partial sums stay few
    const unsigned int nb = (unsigned int)(n * bps);
    if (first) *nparts = (int)std::min<long long>(std::min<long long>(nb, max_parts), 608);
    const unsigned int g = (unsigned int)*nparts;  // the last chunk may be smaller: idle blocks add nothing
    if (ham_only)
      k_constraints<0><<<g, CON_THREADS, 0, s>>>(A, nb, bps, first);
    else if (order == 4)
      k_constraints<2><<<g, CON_THREADS, 0, s>>>(A, nb, bps, first);
    else
      k_constraints<4><<<g, CON_THREADS, 0, s>>>(A, nb, bps, first);
  });
}

cudaError_t launch_psi4(int order, FxWork work, size_t rec_doubles, const double origin[3], const double h[3],
                        double* psi_re, double* psi_im, double* inv_re, double* inv_im, double* E, double* B,
                        unsigned int* flag, cudaStream_t s) {
  WeylArgs A{work,   {origin[0], origin[1], origin[2]}, {h[0], h[1], h[2]}, psi_re, psi_im, inv_re, inv_im, E, B, flag,
             {}};
  first_weights(order, h, A.c1);
  const int bps = (work.one.T.vol + CON_THREADS - 1) / CON_THREADS;
  return through_record(order, work, ham_list(), rec_doubles, s, [&](const FxWork& W, long long n, bool) {
    A.W = W;
    if (order == 4)
      k_psi4<2><<<(unsigned int)(n * bps), CON_THREADS, 0, s>>>(A, bps);
    else
      k_psi4<4><<<(unsigned int)(n * bps), CON_THREADS, 0, s>>>(A, bps);
  });
}

// Chunks of an overlapped stage, about; and the fewest tiles worth it.
constexpr int OVERLAP_CHUNKS = 8;
constexpr long long OVERLAP_MIN_TILES = 608;

// Tiles of a chunk: multiples of 76, so that the algebra warps of 152 SMs take
// equally many 32-point groups each.
static long long overlap_chunk(long long ntiles, long long half) {
  return std::min((ntiles + OVERLAP_CHUNKS - 1) / OVERLAP_CHUNKS + 75, half) / 76 * 76;
}

cudaError_t launch_stage64(int order, const FxWork& work, int vol, long long ntiles, long long slots,
                           const Gauge& gz, const StageOut& out, cudaStream_t s) {
  if (slots < 1) return cudaErrorInvalidValue;
  DerivArgs D{work, rhs_list(), out.in, gz.advect_gauge != 0, gz.lapse == 2, gz.shift == 1, out.mode == 0};
  AlgebraArgs A{work, out};
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (ntiles < OVERLAP_MIN_TILES || slots < 2 * 76) {
    const long long chunks = (ntiles + slots - 1) / slots, per = (ntiles + chunks - 1) / chunks;
    for (long long t = 0; t < ntiles && e == cudaSuccess; t += per) {
      const long long n = std::min(per, ntiles - t);
      D.W.tile0 = A.W.tile0 = work.tile0 + t;
      e = order == 4 ? launch_derivs<4>(D, n, s) : launch_derivs<8>(D, n, s);
      if (e != cudaSuccess) break;
      e = launch_algebra(A, n, vol, 4 * sms, s);
    }
    return e;
  }
  // the record as two halves: the derivatives of one chunk go into one while
  // the algebra reads the chunk before from the other
  const long long half = slots / 2;
  const long long per = overlap_chunk(ntiles, half);
  OverlapArgs O;
  O.groups = (vol + 31) / 32;
  double* const recs[2] = {work.rec, work.rec + half * work.slot};
  long long prev = 0;
  int side = 0;
  for (long long t = 0; t < ntiles && e == cudaSuccess; t += per, side ^= 1) {
    const long long n = std::min(per, ntiles - t);
    D.W.tile0 = work.tile0 + t;
    D.W.rec = recs[side];
    if (t == 0) {
      e = order == 4 ? launch_derivs<4>(D, n, s) : launch_derivs<8>(D, n, s);
    } else {
      O.D = D;
      O.A = A;
      O.nd = (unsigned int)n;
      O.na = (unsigned int)prev;
      e = order == 4 ? launch_overlap<4>(O, sms, s) : launch_overlap<8>(O, sms, s);
    }
    A.W.tile0 = D.W.tile0;
    A.W.rec = D.W.rec;
    prev = n;
  }
  if (e != cudaSuccess) return e;
  return launch_algebra(A, prev, vol, 4 * sms, s);
}

long long stage64_slots(long long ntiles) {
  return ntiles < OVERLAP_MIN_TILES ? ntiles : 2 * overlap_chunk(ntiles, ntiles);
}

long long stage64_launches(long long ntiles, long long slots) {
  if (ntiles < OVERLAP_MIN_TILES || slots < 2 * 76) return 2 * ((ntiles + slots - 1) / slots);
  const long long per = overlap_chunk(ntiles, slots / 2);
  return (ntiles + per - 1) / per + 1;
}

cudaError_t bounds_take_stage64(unsigned long long* out) { return bounds_take_local(out); }

}  // namespace bssn
