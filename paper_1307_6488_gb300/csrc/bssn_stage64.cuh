// The algebra half of the FP64 stage, one point at a time, and the kernel that
// runs it beside the derivatives of the next tiles.
#pragma once
#include "bssn_bounds.cuh"
#include "bssn_fixed.cuh"
#include "bssn_point64.cuh"

namespace bssn {

// Point idx of a tile; false outside the grid.
struct TilePoint {
  int i, j, k;
  long long p;
};
__device__ __forceinline__ bool tile_point(const FxGrid& G, int ti, int tj, int tk, int idx, TilePoint& q) {
  if (idx >= G.T.vol) return false;
  const int yz = idx / G.T.tx;
  q.i = ti * FX_T + idx - yz * G.T.tx;
  q.j = tj * FX_T + yz % G.T.ty;
  q.k = tk * FX_T + yz / G.T.ty;
  if (q.i >= G.L.nx || q.j >= G.L.ny || q.k >= G.L.nz) return false;
  q.p = G.L.off0 + q.i + q.j * G.L.sy + q.k * G.L.sz;
  return in_range(q.p, q.p, padded_points(G.L));
}

// Which variables a call of algebra_point is for: all of them, At_ij, or the
// others (the compiler drops the arithmetic that no stored value needs; At_ij
// takes the Ricci tensor and about half of the instructions).
enum AlgebraPart { PART_ALL = 0, PART_AT = 1, PART_REST = 2 };
template <int PART>
__host__ __device__ constexpr bool in_part(int v) {
  return PART == PART_ALL || (v >= V_AT11 && v <= V_AT33) == (PART == PART_AT);
}

// Point idx of a slot: the pointwise right-hand side from the record of
// k_derivs (with its advection + dissipation sums) and the stage update.
template <int PART>
__device__ __forceinline__ void algebra_point(const FxWork& Wk, const StageOut& S, unsigned int slot, int idx) {
  int ti, tj, tk;
  const FxGrid& G = fx_locate(Wk, Wk.tile0 + slot, ti, tj, tk);
  TilePoint pt;
  if (!tile_point(G, ti, tj, tk, idx, pt)) return;
  const long long p = pt.p, vs = G.L.vs;
  const int vol = G.T.vol;
  const double* __restrict__ rec = Wk.rec + (long long)slot * Wk.slot + idx;
  const double* __restrict__ ys = G.buf[S.in] + p;
  Point64 Q;
#pragma unroll
  for (int v = 0; v < NV; ++v) Q.u[v] = __ldg(ys + v * vs);
  auto r = [&](int o) { return __ldg(rec + o * vol); };
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Q.dW[d] = r(d);
    Q.da[d] = r(9 * 7 + d);
    Q.dK[d] = r(REC_K + d);
#pragma unroll
    for (int s = 0; s < 6; ++s) Q.hg[d][s] = r(9 * (1 + s) + d);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Q.db[d][c] = r(9 * (8 + c) + d);
      Q.hG[d][c] = r(REC_GAM + 3 * c + d);
    }
  }
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    Q.ddW[s] = r(3 + s);
    Q.dda[s] = r(9 * 7 + 3 + s);
#pragma unroll
    for (int c = 0; c < 3; ++c) Q.ddb[c][s] = r(9 * (8 + c) + 3 + s);
#pragma unroll
    for (int c = 0; c < 6; ++c) Q.hgg[c][s] = r(9 * (1 + c) + 3 + s);
  }
  double rhs[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) rhs[v] = r(REC_EXT + v);
  rhs_point64(Q, S.gz, G.C.a, G.C.a2, G.C.ia, G.C.b, rhs);
  if (S.mode == 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (in_part<PART>(v)) S.rhs[v * vs + p] = rhs[v];
    return;
  }
  const RK& rk = S.rk;
  const double* y0 = G.buf[0] + p;  // may be the output: read before it is written
  double* acc = G.buf[3] + p;
  double* out = G.buf[S.out] + p;
  if (rk.method == 3) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (!in_part<PART>(v)) continue;
      const long long o = v * vs;
      out[o] = fma(rk.cdt, rhs[v], fma(rk.a1, Q.u[v], rk.a0 * y0[o]));
    }
    return;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (!in_part<PART>(v)) continue;
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

// Derivatives of one chunk of tiles beside the algebra of the chunk before.
// k_derivs leaves the FP64 pipe mostly idle and k_algebra everything else, so
// each SM runs both at once: one block whose first 16 warps take (tile,
// variable) pairs of chunk D in turn, while the others take 32 points of chunk
// A at a time, neither waiting for the other. How many algebra warps: the
// derivatives of 4th order are less work, so more of the SM goes to the
// algebra (101x93x87, 8th order, RK3 step with 8 / 12 / 16: 8.01 / 8.34 / 9.26
// ms, one kernel after the other 8.67; 32 patches, 4th order: 31.1 / 29.1 /
// 30.9, one after the other 31.4).
template <int P>
constexpr int OVERLAP_THREADS = FX_THREADS + 32 * (P == 4 ? 12 : 8);

struct OverlapArgs {
  DerivArgs D;    // chunk whose derivatives are made
  AlgebraArgs A;  // chunk whose algebra is done
  unsigned int nd, na;   // their slots
  int groups;     // 32-point groups of a slot
};

template <int P>
__global__ void __launch_bounds__(OVERLAP_THREADS<P>, 1) k_overlap(const __grid_constant__ OverlapArgs A) {
  if (threadIdx.x < FX_THREADS) {
    extern __shared__ __align__(16) unsigned char fx_smem[];
    __shared__ unsigned int red[3][FX_THREADS / 32];
    int4* g = (int4*)fx_smem;
    int2* box = (int2*)(g + 3 * FxSmem<P>::GN);
    const DerivArgs& D = A.D;
    const unsigned int items = A.nd * (unsigned int)D.list.n;
    const unsigned int turn = A.nd / (unsigned int)D.list.n;
    for (unsigned int it = blockIdx.x; it < items; it += gridDim.x) {
      // the chunk's tiles from another one on for every variable: a tile that
      // takes long (fx_refine) does so for several, which are not to meet in one
      // block (chunks are multiples of half a round; RK3 at 100^3 11.3 -> 10.4 ms)
      const unsigned int e = it / A.nd;
      unsigned int slot = it - e * A.nd + e * turn;
      if (slot >= A.nd) slot -= A.nd;
      int ti, tj, tk;
      const FxGrid& G = fx_locate(D.W, D.W.tile0 + slot, ti, tj, tk);
      const double* u = G.buf[D.in];
      fx_tile<P>(G.L, G.C, G.T, D.list, (int)e, D.advect_gauge, D.lapse_frozen, D.shift_frozen, D.ko, u,
                 ti, tj, tk, box, g, red, D.W.rec + (long long)slot * D.W.slot);
      fx_sync();  // the next tile reuses the shared memory
    }
  } else {
    constexpr unsigned int WARPS = (OVERLAP_THREADS<P> - FX_THREADS) / 32;
    const unsigned int warp = (threadIdx.x - FX_THREADS) >> 5, n = A.na * (unsigned int)A.groups;
    for (unsigned int q = blockIdx.x * WARPS + warp; q < n; q += gridDim.x * WARPS) {
      const unsigned int slot = q / (unsigned int)A.groups;
      algebra_point<PART_ALL>(A.A.W, A.A.S, slot, (int)(q - slot * A.groups) * 32 + (int)(threadIdx.x & 31));
    }
  }
}

}  // namespace bssn
