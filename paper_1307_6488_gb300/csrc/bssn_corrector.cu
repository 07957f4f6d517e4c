// Learned corrector: a 5-layer 3x3x3 convolutional network (24 -> 32 -> 32
// -> 32 -> 32 -> 24 channels, GELU after the first four layers, output
// added to a coarse RK4 step) with its own BF16 tensor-core training and
// inference kernels on Blackwell tcgen05 (FP32 accumulation in TMEM).
//
// Every layer is padded to 32 input and 32 output channels (the extra input
// channels carry zeros, the extra output channels have zero weights and get
// zero gradients), so one tensor-core shape serves all three convolutions:
//   forward and input-gradient ("dgrad") - an implicit GEMM with M = 128
//     output entries, N = 32 output channels, K = 27 taps x 32 channels. A
//     TMA box brings a whole slab (R + 2 rows of one input plane, all 32
//     channels, chunk-major, unswizzled) into shared memory once; the A
//     operand of each of the 9 in-plane taps is that slab seen through a
//     descriptor shifted by the tap's entry offset, and each slab serves the
//     three output planes it neighbours (k_conv_tc below);
//   weight gradient ("wgrad") - M = 3 dz taps x 32 input channels (+ 32
//     rows of ones: the bias), N = up to 3 dy x 32 output channels, K = points
//     (one x-row per step). Both operands are padded arrays as they are stored:
//     rows of points with 8 channels contiguous are an operand whose
//     contiguous direction is M or N, which the tensor core takes. Each CTA
//     streams a range of rows, keeps all 27 taps' sums in TMEM, and writes a
//     partial, summed afterwards in a fixed order (k_wgrad_rows below).
// Activations are zero outside the box (zero padding); the backward pass is
// its exact adjoint.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/bssn.h"
#include "bssn_common.cuh"
#include "bssn_tc.cuh"

using namespace bssn;

namespace {

constexpr int CH = 32;
constexpr int NL = 5;
constexpr int NTAP = 27;
constexpr int W_TAP_BYTES = CH * CH * 2;  // 2 KB per tap
constexpr int LAYER_PARAMS = NTAP * CH * CH + CH;

struct Geom {
  int S, Z, Y, X;  // samples and interior points per axis
};

// Padded activations and gradients (BF16, one zero point on every side) are
// stored chunk-major: per sample s and padded plane zz (0 .. Z+1), four
// planes of 8 channels each, [Y+2][X+2][8]. Offsets below count 8-channel
// groups (16 bytes). A slab of consecutive rows of one chunk plane is then
// contiguous, which the convolution's shared-memory slabs rely on.
__host__ __device__ inline long long chunk_off(const Geom& G, int s, int zz, int q, int yy, int xx) {
  return ((((long long)s * (G.Z + 2) + zz) * 4 + q) * (G.Y + 2) + yy) * (G.X + 2) + xx;
}
// A slab's copy takes a row's points as one dimension, in 8-byte elements,
// where a box may be that wide (256 elements): runs of a whole row instead of
// 16 bytes (inference at 64^3 160 -> 157 us, a training step 2.29 -> 2.24 ms).
__host__ __device__ inline bool slab_rows(int X) { return 2 * (X + 1) <= 256; }
__host__ __device__ inline long long chunk_stride(const Geom& G) { return (long long)(G.Y + 2) * (G.X + 2); }

// the 32 channels (4 x 16 bytes) of interior point (s, z, y, x)
__device__ __forceinline__ void store_point(const Geom& G, __nv_bfloat16* buf, int s, int z, int y, int x,
                                            const __nv_bfloat16* h) {
  uint4* p = (uint4*)buf + chunk_off(G, s, z + 1, 0, y + 1, x + 1);
  const long long cs = chunk_stride(G);
#pragma unroll
  for (int q = 0; q < 4; ++q) p[q * cs] = ((const uint4*)h)[q];
}

// The activation: the tanh form of GELU (Hendrycks and Gimpel 2016),
// x (1 + tanh u) / 2 with u = sqrt(2/pi) (x + 0.044715 x^3), on the hardware
// tanh (tanh.approx.f32, relative error ~2^-11, far below the BF16 rounding
// of the stored activation); a few instructions against ~25 for erff.
__device__ __forceinline__ float tanh_hw(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gelu_f(float x) {
  const float u = 0.7978845608028654f * fmaf(0.044715f * x, x * x, x);
  return 0.5f * x * (1.f + tanh_hw(u));
}
__device__ __forceinline__ float gelu_grad_f(float x) {
  const float u = 0.7978845608028654f * fmaf(0.044715f * x, x * x, x);
  const float t = tanh_hw(u);
  const float du = 0.7978845608028654f * fmaf(0.134145f * x, x, 1.f);
  return 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * du;
}

// ---------------------------------------------------------------- forward / dgrad
// MODE 0: out = conv(a) + bias; zout (FP32, unpadded) and act_out (BF16,
//         padded, GELU applied if gelu) as requested.
// MODE 1: d = conv(g) with the transposed, flipped weights; if zprev, d *=
//         GELU'(zprev); act_out (BF16, padded) receives d.
//
// Shared-memory slabs instead of one load per tap. A work unit is (sample,
// block of R output rows, run of L output planes). For every input plane the
// unit needs (L + 2 of them) one TMA box brings rows y0-1 .. y0+R, points
// x = 0 .. X (the last one is the zero pad) and all 32 channels into a slab
// laid out [chunk of 8 channels][row][x] with X+1 entries per row, so entry
// e = row (X+1) + x sits at e * 16 bytes within its chunk. Because the pad
// entry separates the rows, the input of tap (dy, dx) for output entry e is
// entry e + dy (X+1) + dx: a plain shift. The M = 128 rows of an MMA are 128
// consecutive output entries (pad entries and rows past R give results that
// are discarded), the A operand of every tap is the same slab seen through a
// shifted no-swizzle descriptor (core matrices 8 entries x 16 bytes, SBO =
// 128 bytes, LBO = one chunk), and T tiles of 128 entries cover the R rows.
//
// The three dz taps share their A operand. Input plane i feeds output planes
// i + 1, i and i - 1 through the weights of dz = 0, 1, 2, so one MMA with N =
// 96 (the three dz blocks of one in-plane tap stacked along N; the weights sit
// in shared memory as [dy dx][dz][32 co][32 ci]) adds all three
// contributions, each into its own output plane's accumulator. TMEM holds, per
// tile, K blocks of 32 columns; output plane z0 + q of a unit accumulates in
// block L - 1 - q, so the blocks of planes i + 1, i, i - 1 are adjacent and in
// dz order. At the unit's first and last two input planes fewer outputs lie
// in the unit and the MMA narrows to N = 32 or 64. Every MMA accumulates:
// the epilogue writes zeros into a block when it has read it (and into every
// block at the start), before handing it back.
//   warp 16 (one lane) loads the 27 weight taps once and streams slabs into a
//                      4-deep ring;
//   warp 17            issues 9 taps x 2 MMAs (K = 16) per tile and input
//                      plane (the whole warp runs the loop, one elected lane
//                      issues), releases the slab when they finish and hands
//                      a block to the epilogue after its last contribution;
//                      it never waits for an MMA to finish;
//   warps 0-15         read the accumulators out (warp w: TMEM lanes
//                      32 (w % 4) .. +31, channels 8 (w / 4) .. +7), run the
//                      epilogue and zero the block; four warps per lane
//                      quarter keep enough loads and stores in flight.
// Every wait is bounded; a role that times out sets the error word and the
// CTA-wide abort flag, the others leave their loops, in-flight copies and
// MMAs are waited for (bounded) and TMEM is freed.
// Resident convolution CTAs per SM. One (the default) holds all of TMEM,
// four slabs and 16 epilogue warps. Two (each with half of TMEM, two slabs
// and 8 epilogue warps, so that one CTA's barrier hand-offs overlap the
// other's MMAs) measured slower: 0.25 against 0.19-0.20 ms for a 64^3
// single-sample forward pass.
#ifndef CONV_CTAS_PER_SM
#define CONV_CTAS_PER_SM 1
#endif
constexpr int CONV_CTAS = CONV_CTAS_PER_SM;
constexpr int EPI_WARPS = CONV_CTAS == 2 ? 8 : 16;
constexpr int CONV_THREADS = 32 * (EPI_WARPS + 2);
constexpr int WG_THREADS = 192;
constexpr int SLABS = CONV_CTAS == 2 ? 2 : 4;
constexpr int KMAX = CONV_CTAS == 2 ? 8 : 16;  // accumulator blocks per tile at T = 1 (this CTA's TMEM columns / 32)
// dynamic shared memory per CTA: at most what CONV_CTAS CTAs per SM can have,
// at least enough that no further CTA fits beside them (the TMEM would not)
constexpr int CONV_SMEM_MAX = CONV_CTAS == 2 ? 115712 : 232448;
constexpr int CONV_SMEM_MIN = CONV_CTAS == 2 ? 79872 : 118784;

struct ConvPlan {
  int R;              // output rows per unit
  int T;              // 128-entry M tiles covering R rows of X+1 entries
  int K;              // accumulator blocks (of 32 columns) per tile: the most planes a unit may have
  int L;              // output planes per unit (set per call, <= K)
  int nyb, nzs;       // row blocks, plane runs
  int chunk_bytes;    // (R+2)(X+1) x 16
  int plane_bytes;    // 4 chunks
  int slab_stride;    // plane_bytes rounded up to 128 (TMA destinations are 128-byte aligned)
  int tail_bytes;     // past the last slab: reads of discarded rows
  int tmem_cols;      // power of two >= T K 32
  int smem;           // dynamic shared memory
  int slab_off;       // offset of slab 0 from the 1024-aligned base
  int bar_off;        // offset of the barriers
};

// 8 channels (one 16-byte chunk, channels 8 q .. 8 q + 7) of interior point (s, z, y, x)
__device__ __forceinline__ void store_chunk(const Geom& G, __nv_bfloat16* buf, int s, int z, int y, int x, int q,
                                            const __nv_bfloat16* v) {
  *((uint4*)buf + chunk_off(G, s, z + 1, q, y + 1, x + 1)) = *(const uint4*)v;
}

template <int MODE>
__global__ void __launch_bounds__(CONV_THREADS, CONV_CTAS)
    k_conv_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, Geom G, ConvPlan P,
              const float* __restrict__ bias, float* __restrict__ zout, __nv_bfloat16* __restrict__ act_out,
              const float* __restrict__ zprev, int gelu, unsigned int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* Wt = base;                // [9 (dy, dx)][3 dz][32 co][32 ci], 64-byte swizzle
  uint8_t* slab = base + P.slab_off;  // SLABS x slab_stride; the 16 bytes before it are zero
  uint64_t* bars = (uint64_t*)(base + P.bar_off);
  uint64_t* full = bars;
  uint64_t* empty = bars + SLABS;
  uint64_t* tfull = bars + 2 * SLABS;   // [KMAX] block complete
  uint64_t* tempty = tfull + KMAX;      // [KMAX] block read out and zeroed (one arrive per epilogue warp)
  uint64_t* wbar = tempty + KMAX;
  uint64_t* drain = wbar + 1;           // all MMAs of this CTA finished
  uint32_t* tslot = (uint32_t*)(drain + 1);
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int XS = G.X + 1;
  const int units = G.S * P.nyb * P.nzs;
  auto unit_pos = [&](int u, int& s, int& yb, int& z0, int& len) {
    const int zs = u % P.nzs;
    const int t = u / P.nzs;
    yb = t % P.nyb;
    s = t / P.nyb;
    z0 = zs * P.L;
    len = min(P.L, G.Z - z0);
  };

  // zero the entry before slab 0, the gap after each slab (its last entry is
  // the entry before the next slab: the x = -1 pad of tap dx = -1 at the
  // first output entry) and the tail (read only for discarded rows)
  {
    uint32_t* lead = (uint32_t*)(slab - 128);
    if (tid < 32) lead[tid] = 0u;
    const int gap = P.slab_stride - P.plane_bytes;
    for (int i = tid; i < SLABS * (gap / 4); i += blockDim.x)
      ((uint32_t*)(slab + (i / (gap / 4)) * P.slab_stride + P.plane_bytes))[i % (gap / 4)] = 0u;
    uint32_t* tail = (uint32_t*)(slab + SLABS * P.slab_stride);
    for (int i = tid; i < P.tail_bytes / 4; i += blockDim.x) tail[i] = 0u;
    tc::fence_proxy_async();
  }
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < SLABS; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int b = 0; b < KMAX; ++b) {
      tc::mbar_init(&tfull[b], 1);
      tc::mbar_init(&tempty[b], EPI_WARPS);
    }
    tc::mbar_init(wbar, 1);
    tc::mbar_init(drain, 1);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(tslot, (uint32_t)P.tmem_cols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = *tslot;
  const bool any = (int)blockIdx.x < units;
  const uint32_t tile_cols = (uint32_t)(P.K * 32);
  // the next layer may be scheduled onto SMs as this grid's CTAs leave them
  if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == EPI_WARPS) {
    // ---- TMA producer
    if (lane == 0 && any) {
      tc::mbar_expect_tx(wbar, NTAP * W_TAP_BYTES);
      // tap k = 9 dz + 3 (dy + 1) + (dx + 1) goes to slot 3 (k % 9) + k / 9
      for (int k = 0; k < NTAP; ++k)
        tc::tma_load_2d(Wt + (3 * (k % 9) + k / 9) * W_TAP_BYTES, &tmW, 0, k * CH, wbar);
      // launched as a programmatic dependent of the previous layer: everything
      // above overlapped its tail; its output is read only from here on (a
      // no-op for an ordinary launch)
      asm volatile("griddepcontrol.wait;" ::: "memory");
      uint32_t g = 0;  // slabs issued (sequence over all units)
      bool ok = true;
      for (int u = blockIdx.x; ok && u < units; u += gridDim.x) {
        int s, yb, z0, len;
        unit_pos(u, s, yb, z0, len);
        for (int k = 0; k < len + 2; ++k) {
          const uint32_t buf = g % SLABS;
          if (g >= SLABS && !tc::mbar_wait_or_abort(&empty[buf], ((g / SLABS) - 1) & 1, &abort_flag)) {
            if (!abort_flag) atomicOr(err, 1u);
            abort_flag = 1;
            ok = false;
            break;
          }
          tc::mbar_expect_tx(&full[buf], (uint32_t)P.plane_bytes);
          // padded plane z0 + k holds input plane z0 - 1 + k; padded row yb R
          // is output row yb R - 1
          if (slab_rows(G.X))
            tc::tma_load_4d(slab + buf * P.slab_stride, &tmA, 2, yb * P.R, 0, s * (G.Z + 2) + z0 + k, &full[buf]);
          else
            tc::tma_load_5d(slab + buf * P.slab_stride, &tmA, 0, 1, yb * P.R, 0, s * (G.Z + 2) + z0 + k, &full[buf]);
          ++g;
        }
      }
      // the last use of every slab buffer has landed before the CTA leaves
      for (uint32_t q = g > SLABS ? g - SLABS : 0; q < g; ++q)
        (void)tc::mbar_wait(&full[q % SLABS], (q / SLABS) & 1, 100000000ull);
      (void)tc::mbar_wait(wbar, 0, 100000000ull);
    }
  } else if (warp == EPI_WARPS + 1) {
    // ---- MMA issuer: the whole warp runs the loop on warp-uniform
    // descriptors and one elected lane issues each MMA and commit
    if (any) {
      bool ok = tc::warp_wait_or_abort(wbar, 0, &abort_flag);
      const uint32_t slab0 = tc::smem_u32(slab);
      const uint64_t w_desc0 = tc::smem_desc(tc::smem_u32(Wt), 16, 512, tc::SWZ_64B);
      constexpr uint32_t IDESC32 = tc::idesc_bf16_f32(128, 32), IDESC64 = tc::idesc_bf16_f32(128, 64),
                         IDESC96 = tc::idesc_bf16_f32(128, 96);
      const uint32_t k_half = (uint32_t)(2 * P.chunk_bytes) >> 4;
      uint32_t g = 0;  // slab sequence at the unit's first input plane
      uint32_t use = 0;  // units done: each unit uses every block once
      for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++use) {
        int s, yb, z0, len;
        unit_pos(u, s, yb, z0, len);
        const uint32_t par = use & 1;
        for (int k = 0; ok && k < len + 2; ++k) {
          // input plane z0 - 1 + k feeds output planes q = k - dz (dz = 0, 1, 2)
          // of the unit that exist: q_lo .. q_hi
          const int q_hi = min(len - 1, k), q_lo = max(0, k - 2);
          const int n = q_hi - q_lo + 1;
          const int dz0 = k - q_hi;
          // the first contribution to plane q = k: its block must be empty
          if (k < len && !tc::warp_wait_or_abort(&tempty[P.L - 1 - k], par, &abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t gg = g + (uint32_t)k;
          const uint32_t buf = gg % SLABS;
          if (!tc::warp_wait_or_abort(&full[buf], (gg / SLABS) & 1, &abort_flag)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          // descriptors change only in the start-address field (bits 0-13,
          // bytes / 16): tap (dy, dx) shifts A by (1 + dy)(X+1) + dx entries,
          // the second K half adds two chunks (A) or 32 bytes (B), the next
          // tap's weights add 6 KB and the next dz block 2 KB
          const uint64_t a_plane =
              tc::smem_desc(slab0 + buf * (uint32_t)P.slab_stride, (uint32_t)P.chunk_bytes, 128, tc::SWZ_NONE);
          const uint64_t b_plane = w_desc0 + (uint64_t)(dz0 * (W_TAP_BYTES >> 4));
          const uint32_t idesc = n == 3 ? IDESC96 : (n == 2 ? IDESC64 : IDESC32);
          const uint32_t dcol = (uint32_t)(32 * (P.L - 1 - q_hi));
          for (int j = 0; j < P.T; ++j) {
            const uint64_t a_tile = a_plane + (uint64_t)(128 * j) - 1;  // 128 entries (of 16 bytes) per tile
            const uint32_t d = taddr + (uint32_t)j * tile_cols + dcol;
#pragma unroll
            for (int t = 0; t < 9; ++t) {
              const uint64_t a_tap = a_tile + (uint64_t)(XS * (t / 3) + (t % 3));
#pragma unroll
              for (int kk = 0; kk < 2; ++kk)
                tc::mma_bf16_elect(d, a_tap + (uint64_t)(kk * k_half),
                                   b_plane + (uint64_t)(t * (3 * W_TAP_BYTES >> 4) + 2 * kk), idesc, 1u);
            }
          }
          tc::mma_commit_elect(&empty[buf]);  // the slab is free once these MMAs finish
          // plane q = k - 2 has had its last contribution
          if (k >= 2) tc::mma_commit_elect(&tfull[P.L - 1 - (k - 2)]);
        }
        // planes past the end of the grid (a short last run) are handed over
        // empty so that every block completes once per unit
        for (int q = len; ok && q < P.L; ++q) {
          if (!tc::warp_wait_or_abort(&tempty[P.L - 1 - q], par, &abort_flag)) {
            ok = false;
            break;
          }
          tc::mma_commit_elect(&tfull[P.L - 1 - q]);
        }
        g += (uint32_t)(len + 2);
      }
      if (!ok && lane == 0) {
        if (!abort_flag) atomicOr(err, 1u);
        abort_flag = 1;
      }
      // every MMA this warp issued has finished before TMEM is freed
      tc::mma_commit_elect(drain);
      (void)tc::warp_wait(drain, 0, 100000000ull);
    }
  } else {
    // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 and the
    // 8-channel chunks cq0 + i EPI_WARPS/4 (i < CPW) of the 4
    constexpr int CPW = 16 / EPI_WARPS;
    const int cq0 = warp >> 2;
    const uint32_t lane_base = taddr + ((uint32_t)((warp & 3) * 32) << 16);
    float bq[CPW][8];
#pragma unroll
    for (int i = 0; i < CPW; ++i)
#pragma unroll
      for (int c = 0; c < 8; ++c) bq[i][c] = MODE == 0 ? __ldg(bias + 8 * (cq0 + i * (EPI_WARPS / 4)) + c) : 0.f;
    // every block starts zeroed and empty
    for (int j = 0; j < P.T; ++j)
      for (int b = 0; b < P.K; ++b)
#pragma unroll
        for (int i = 0; i < CPW; ++i)
          tc::tmem_st8_zero(lane_base + (uint32_t)j * tile_cols + (uint32_t)(32 * b + 8 * (cq0 + i * (EPI_WARPS / 4))));
    tc::tmem_wait_st();
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0)
      for (int b = 0; b < P.K; ++b) tc::mbar_arrive(&tempty[b]);
    uint32_t use = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < units; u += gridDim.x, ++use) {
      int s, yb, z0, len;
      unit_pos(u, s, yb, z0, len);
      for (int q = 0; q < P.L; ++q) {
        const int b = P.L - 1 - q;
        ok = tc::mbar_wait_or_abort(&tfull[b], use & 1, &abort_flag);
        ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-collective
        if (!ok) {
          if (lane == 0) {
            if (!abort_flag) atomicOr(err, 2u);
            abort_flag = 1;
          }
          break;
        }
        tc::fence_after_sync();
        const int z = z0 + q;
        for (int j = 0; q < len && j < P.T; ++j) {
          float acc[CPW][8];
#pragma unroll
          for (int i = 0; i < CPW; ++i) {
            const uint32_t col = lane_base + (uint32_t)j * tile_cols +
                                 (uint32_t)(32 * b + 8 * (cq0 + i * (EPI_WARPS / 4)));
            tc::tmem_ld8(col, acc[i]);
            tc::tmem_st8_zero(col);
          }
          const int e = XS + 128 * j + 32 * (warp & 3) + lane;
          const int row = e / XS, x = e - row * XS;
          const int y = yb * P.R + row - 1;
          if (x >= G.X || row > P.R || y >= G.Y) continue;
          const long long pt = (((long long)s * G.Z + z) * G.Y + y) * G.X + x;
#pragma unroll
          for (int i = 0; i < CPW; ++i) {
            const int cq = cq0 + i * (EPI_WARPS / 4);
            float* a = acc[i];
            __align__(16) __nv_bfloat16 hv[8];
            if (MODE == 0) {
#pragma unroll
              for (int c = 0; c < 8; ++c) a[c] += bq[i][c];
              if (zout) {
                float4* zo = (float4*)(zout + pt * CH + 8 * cq);
                zo[0] = make_float4(a[0], a[1], a[2], a[3]);
                zo[1] = make_float4(a[4], a[5], a[6], a[7]);
              }
              if (act_out) {
#pragma unroll
                for (int c = 0; c < 8; ++c) hv[c] = __float2bfloat16_rn(gelu ? gelu_f(a[c]) : a[c]);
                store_chunk(G, act_out, s, z, y, x, cq, hv);
              }
            } else {
              if (zprev) {
                const float4* zp = (const float4*)(zprev + pt * CH + 8 * cq);
#pragma unroll
                for (int q4 = 0; q4 < 2; ++q4) {
                  const float4 v = __ldg(zp + q4);
                  a[4 * q4] *= gelu_grad_f(v.x);
                  a[4 * q4 + 1] *= gelu_grad_f(v.y);
                  a[4 * q4 + 2] *= gelu_grad_f(v.z);
                  a[4 * q4 + 3] *= gelu_grad_f(v.w);
                }
              }
#pragma unroll
              for (int c = 0; c < 8; ++c) hv[c] = __float2bfloat16_rn(a[c]);
              store_chunk(G, act_out, s, z, y, x, cq, hv);
            }
          }
        }
        // zeros written, then the block goes back to the MMA warp
        tc::tmem_wait_st();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&tempty[b]);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(taddr, (uint32_t)P.tmem_cols);
}

// ---------------------------------------------------------------- wgrad
// dW[t][co][ci] = sum over points p of act(p + off_t, ci) g(p, co): per CTA a
// range of output x-rows (s, z, y), all 27 taps at once.
//   The CTA steps through the activation rows y' that its output rows of a
//   plane reach (one more on each side). A step loads the row's three dz
//   planes, X + 2 points each, and the gradient row y = y' where there is
//   one; row y' meets the gradient rows y' - dy, three of them (fewer at the
//   ends).
//   In shared memory a box is [chunk of 8 channels][point][8 channels], no
//   swizzle: 8 points x 8 channels are one 128-byte core matrix with the
//   channels contiguous (M- and N-major operands), the next 8 points follow
//   (leading offset 128 bytes), the next 8 channels are a chunk further
//   (stride offset). The three dz boxes and a box of ones lie together: M = 128 rows
//   (dz, ci) and 32 rows whose sums are the bias gradient; a shift dx is 16
//   bytes of the start address. Gradient rows lie together too, so N is up to 3 x
//   32 (y, co); K = the row's XW points. Per shift 96 TMEM columns sum over
//   the rows, in row order for every tap.
//   A copy of the operands channels-first, once per shift, had cost 20 passes
//   of 25 us in a training step at 64^3, batch 4 (2.98 -> 2.29 ms without).
//   Loading each shift of each row and N = 32 per MMA, a step moved 40 KB and
//   read the M operand from shared memory nine times (168 us per layer);
//   now 17 KB and three times (57 us; the training step 2.24 -> 1.68 ms).
//   warp 4 (one lane) streams the rows; warp 5 (whole warp, one elected lane)
//   issues 3 x XW/16 MMAs per step; warps 0-2 write the 27 taps' partial sums
//   at the end, warp 3 the bias gradient's.
constexpr int WR_Y = 6;         // activation rows in the ring
constexpr int WR_B = WR_Y + 2;  // gradient rows in the ring: a row is last read two steps after its own, so
                                // the free slot of an activation row implies the free slot of a gradient row
template <int XW>
struct WR {
  static constexpr int CS = 16 * (XW + 2);               // one chunk of 8 channels of an activation row
  static constexpr int ABOX = 4 * CS;                    // one plane of an activation row
  static constexpr int ROW = 4 * ABOX;                   // three planes and the ones
  static constexpr int GCS = 16 * XW, GBOX = 4 * GCS;    // gradient row
  // the first two gradient slots are held a second time behind the last, so
  // that three rows always lie together
  static constexpr int SMEM = 1024 + WR_Y * ROW + (WR_B + 2) * GBOX + 256;
  static constexpr uint32_t LBO = 8 * 16;                // 8 points
  static constexpr int KSTEPS = XW / 16, KSTEP = 16 * 16 / 16;  // descriptor units (16 bytes) of 16 points
  static_assert(ABOX % 128 == 0 && GBOX % 128 == 0, "TMA destinations stay 128-byte aligned");
};

template <int XW>
__global__ void __launch_bounds__(WG_THREADS, 1)
    k_wgrad_rows(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG, Geom G,
                 int rows_per_cta, float* __restrict__ partial, unsigned int* err) {
  using W = WR<XW>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* Ast = base;                     // [WR_Y][dz, ones] boxes
  uint8_t* Bst = base + WR_Y * W::ROW;     // [WR_B + 2] gradient rows
  uint64_t* bars = (uint64_t*)(Bst + (WR_B + 2) * W::GBOX);
  uint64_t* full = bars;                   // [WR_Y] a step's copies landed
  uint64_t* empty = full + WR_Y;           // [WR_Y] a step's MMAs done
  uint64_t* done = empty + WR_Y;
  uint32_t* tslot = (uint32_t*)(done + 1);
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long total_rows = (long long)G.S * G.Z * G.Y;
  const long long r0 = (long long)blockIdx.x * rows_per_cta;
  const int nrows = (int)(r0 >= total_rows ? 0 : (total_rows - r0 < rows_per_cta ? total_rows - r0 : rows_per_cta));

  for (int i = tid; i < WR_Y * (W::ABOX / 4); i += blockDim.x) {
    const int slot = i / (W::ABOX / 4), q = i % (W::ABOX / 4);
    ((uint32_t*)(Ast + slot * W::ROW + 3 * W::ABOX))[q] = 0x3F803F80u;  // BF16 1.0 pairs
  }
  tc::fence_proxy_async();
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < WR_Y; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(done, 1);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(tslot, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = *tslot;
  if (warp < 4) {  // the sums start at zero: a step adds to one, two or three rows' columns at once
#pragma unroll 1
    for (int c = 0; c < 288; c += 8) tc::tmem_st8_zero(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)c);
    tc::tmem_wait_st();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  constexpr uint32_t MN_MAJOR = (1u << 15) | (1u << 16);  // both operands stored along K, channels contiguous

  if (warp == 4) {
    // ---- TMA producer
    if (lane == 0 && nrows > 0) {
      int e = 0;  // steps issued
      bool ok = true;
      for (int k = 0; ok && k < nrows;) {  // plane by plane: rows ya .. yb-1 of (s, z), the CTA's rows k ..
        const long long R = r0 + k;
        const int ya = (int)(R % G.Y);
        const int yb = G.Y - ya < nrows - k ? G.Y : ya + nrows - k;
        const long long rz = R / G.Y;
        const int zp = (int)(rz / G.Z) * (G.Z + 2) + (int)(rz % G.Z);  // padded plane of dz = -1
        for (int yp = ya; yp < yb + 2; ++yp, ++e) {
          const int sl = e % WR_Y;
          if (e >= WR_Y && !tc::mbar_wait_or_abort(&empty[sl], ((e / WR_Y) - 1) & 1, &abort_flag)) {
            ok = false;
            break;
          }
          const int gs = (k + yp - ya) % WR_B;
          const int copies = yp < yb ? (gs < 2 ? 2 : 1) : 0;
          tc::mbar_expect_tx(&full[sl], (uint32_t)(3 * W::ABOX + copies * W::GBOX));
          // padded row yp holds activation row yp - 1
#pragma unroll
          for (int dz = 0; dz < 3; ++dz)
            tc::tma_load_4d(Ast + sl * W::ROW + dz * W::ABOX, &tmX, 0, yp, zp + dz, 0, &full[sl]);
          for (int c = 0; c < copies; ++c)
            tc::tma_load_4d(Bst + (gs + c * WR_B) * W::GBOX, &tmG, 2, yp + 1, zp + 1, 0, &full[sl]);
        }
        k += yb - ya;
      }
      if (!ok) {
        if (!abort_flag) atomicOr(err, 4u);
        abort_flag = 1;
      }
      // every copy has landed before the CTA leaves
      for (int q = e > WR_Y ? e - WR_Y : 0; q < e; ++q) (void)tc::mbar_wait(&full[q % WR_Y], (q / WR_Y) & 1, 100000000ull);
    }
  } else if (warp == 5) {
    // ---- MMA issuer (warp-uniform, one elected lane issues)
    if (nrows > 0) {
      bool ok = true;
      int e = 0;
      for (int k = 0; ok && k < nrows;) {
        const int ya = (int)((r0 + k) % G.Y);
        const int yb = G.Y - ya < nrows - k ? G.Y : ya + nrows - k;
        for (int yp = ya; yp < yb + 2; ++yp, ++e) {
          const int sl = e % WR_Y;
          if (!tc::warp_wait_or_abort(&full[sl], (e / WR_Y) & 1, &abort_flag)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          // gradient rows ylo .. yhi meet this row; row yp - 2 + c has columns 32 c ..
          const int ylo = yp - 2 > ya ? yp - 2 : ya, yhi = yp < yb ? yp : yb - 1;
          const int n = yhi - ylo + 1;
          const uint32_t idesc = tc::idesc_bf16_f32(128, 32 * n) | MN_MAJOR;
          const uint64_t bd = tc::smem_desc(tc::smem_u32(Bst + (k + ylo - ya) % WR_B * W::GBOX), W::LBO, W::GCS,
                                            tc::SWZ_NONE);
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {
            const uint64_t ad =
                tc::smem_desc(tc::smem_u32(Ast + sl * W::ROW + dx * 16), W::LBO, W::CS, tc::SWZ_NONE);
            const uint32_t d = taddr + (uint32_t)(dx * 96 + (ylo - yp + 2) * 32);
#pragma unroll
            for (int j = 0; j < W::KSTEPS; ++j)
              tc::mma_bf16_elect(d, ad + W::KSTEP * j, bd + W::KSTEP * j, idesc, 1u);
          }
          tc::mma_commit_elect(&empty[sl]);
        }
        k += yb - ya;
      }
      if (!ok && lane == 0) {
        if (!abort_flag) atomicOr(err, 4u);
        abort_flag = 1;
      }
      // completes once every MMA issued above has finished (also on abort)
      tc::mma_commit_elect(done);
    }
  }
  // ---- epilogue (warps 0-2: TMEM lanes 32 w .. = input channels of dz = w - 1;
  // warp 3: the bias gradient, the lanes of the ones, any shift and row)
  bool ok = false;
  if (warp < 4 && nrows > 0) {
    ok = tc::mbar_wait(done, 0);
    if (!ok && lane == 0) atomicOr(err, 8u);
    ok = ok && !abort_flag;
    ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-collective
  }
  tc::fence_after_sync();
  if (warp < 3) {
    for (int g = 0; g < 9; ++g) {
      const int dx = g / 3, dy = 2 - g % 3, t = warp * 9 + dy * 3 + dx;
      // partial[b][t][co][ci]: lane = ci, so each co is one coalesced 128-byte row
      float* out = partial + ((long long)blockIdx.x * NTAP + t) * CH * CH + lane;
      float acc[32];
      if (ok) {
        tc::tmem_ld32(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)(g * 32), acc);
      } else {
#pragma unroll
        for (int co = 0; co < 32; ++co) acc[co] = 0.f;
      }
#pragma unroll
      for (int co = 0; co < 32; ++co) out[co * CH] = acc[co];
    }
  } else if (warp == 3) {
    float acc[32];
    if (ok) {
      tc::tmem_ld32(taddr + ((uint32_t)(3 * 32) << 16), acc);
    } else {
#pragma unroll
      for (int co = 0; co < 32; ++co) acc[co] = 0.f;
    }
    // after the gridDim.x x 27 x 32 x 32 weight partials: gridDim.x x 32 bias partials
    float* out = partial + (long long)gridDim.x * NTAP * CH * CH + (long long)blockIdx.x * CH;
    if (lane == 0)
#pragma unroll
      for (int co = 0; co < 32; ++co) out[co] = acc[co];
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(taddr, 512);
}

// dW[t][co][ci] = sum_b partial[b][t][co][ci] and db[co] = sum_b
// bias_partial[b][co] (db follows dW in the layer's parameters), in a fixed
// order: a block of 8 warps takes 32 consecutive outputs (one per lane,
// coalesced), warp w sums the partials b = w, w + 8, ... in double precision,
// then the 8 warp sums are added in warp order.
__global__ void __launch_bounds__(256) k_wgrad_reduce(const float* __restrict__ partial, int nb,
                                                      float* __restrict__ dW) {
  __shared__ double part[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int idx = blockIdx.x * 32 + lane;  // over 27*32*32 + 32
  double s = 0.0;
  // the loads of several partials ahead of their sums
  if (idx < NTAP * CH * CH) {
#pragma unroll 10
    for (int b = w; b < nb; b += 8) s += partial[(long long)b * NTAP * CH * CH + idx];
  } else if (idx < NTAP * CH * CH + CH) {
    const float* bp = partial + (long long)nb * NTAP * CH * CH + (idx - NTAP * CH * CH);
    for (int b = w; b < nb; b += 8) s += bp[(long long)b * CH];
  }
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && idx < NTAP * CH * CH + CH) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) t += part[q][lane];
    dW[idx] = (float)t;
  }
}

// Unpadded BF16 [pts][32] -> interior of a padded buffer.
__global__ void k_pad_copy(Geom G, const __nv_bfloat16* __restrict__ in, __nv_bfloat16* __restrict__ out) {
  const long long pts = (long long)G.S * G.Z * G.Y * G.X;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y);
    const long long r2 = r / G.Y;
    const int z = (int)(r2 % G.Z), s = (int)(r2 / G.Z);
    store_point(G, out, s, z, y, x, in + i * CH);
  }
}

// Loss: mean over points and the first nout channels of (out - target)^2;
// the gradient 2 (out - target) / (pts nout) goes to g (padded BF16, zero in
// the other channels). Per-block partial sums of squares in part.
// Targets as FP32 points of all samples, or (TargetsBf16) as the samples'
// BF16 pointers, 16-byte aligned: a training step's targets are read where
// they are. Two blocks of 512 threads on each SM: a thread's loads lie 128
// bytes from its neighbour's, so it takes many lines in flight.
struct TargetsF32 {
  const float* p;
  __device__ __forceinline__ void get(long long i, int, long long, float (&t)[CH]) const {
#pragma unroll
    for (int q = 0; q < CH / 4; ++q) ((float4*)t)[q] = __ldg((const float4*)(p + i * CH) + q);
  }
};
struct TargetsBf16 {
  const __nv_bfloat16* p[64];
  __device__ __forceinline__ void get(long long i, int s, long long per_sample, float (&t)[CH]) const {
    const uint4* src = (const uint4*)(p[s] + (i - s * per_sample) * CH);
#pragma unroll
    for (int q = 0; q < CH / 8; ++q) {
      const uint4 v = __ldg(src + q);
      const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        t[8 * q + 2 * c] = __uint_as_float(w[c] << 16);
        t[8 * q + 2 * c + 1] = __uint_as_float(w[c] & 0xFFFF0000u);
      }
    }
  }
};
constexpr int MSE_BLOCKS = 304, MSE_THREADS = 512;  // two blocks on each of 152 SMs

template <typename Targets>
__global__ void __launch_bounds__(MSE_THREADS)
    k_mse(Geom G, int nout, const float* __restrict__ out, const __grid_constant__ Targets target,
          __nv_bfloat16* __restrict__ g, double* __restrict__ part) {
  const long long pts = (long long)G.S * G.Z * G.Y * G.X;
  const float gscale = (float)(2.0 / ((double)pts * nout));  // d loss / d out = 2 (out - target) / (pts nout)
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y);
    const long long r2 = r / G.Y;
    const int z = (int)(r2 % G.Z), s = (int)(r2 / G.Z);
    __align__(16) float o[CH], t[CH];
#pragma unroll
    for (int q = 0; q < CH / 4; ++q) {
      ((float4*)o)[q] = __ldg((const float4*)(out + i * CH) + q);
    }
    target.get(i, s, (long long)G.Z * G.Y * G.X, t);
    __align__(16) __nv_bfloat16 h[32];
    float sq = 0.f;  // this point's sum of squares (at most 32 terms)
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      float gv = 0.f;
      if (c < nout) {
        const float d = o[c] - t[c];
        sq = fmaf(d, d, sq);
        gv = d * gscale;
      }
      h[c] = __float2bfloat16_rn(gv);
    }
    acc += (double)sq;
    store_point(G, g, s, z, y, x, h);
  }
  __shared__ double sh[MSE_THREADS];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// FP32 master weights of one layer -> BF16 forward layout [t][co][ci] and
// backward (transposed, flipped) layout [26 - t][ci][co].
__global__ void k_weights_bf16(const float* __restrict__ W, __nv_bfloat16* __restrict__ wf,
                               __nv_bfloat16* __restrict__ wb) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= NTAP * CH * CH) return;
  W += (size_t)blockIdx.y * LAYER_PARAMS;  // layer
  wf += (size_t)blockIdx.y * NTAP * CH * CH;
  wb += (size_t)blockIdx.y * NTAP * CH * CH;
  const int t = idx / (CH * CH), co = (idx / CH) % CH, ci = idx % CH;
  const __nv_bfloat16 v = __float2bfloat16_rn(W[idx]);
  wf[idx] = v;
  wb[((NTAP - 1 - t) * CH + ci) * CH + co] = v;
}

// Adam (decoupled from any weight decay), FP32 master parameters.
__global__ void k_adam(int n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// State (FP64, solver layout) -> network input: channel v = (u_v - off_v) * scale_v
// for v < 24, zero for 24..31; interior of the padded BF16 activation, sample s.
__global__ void k_pack_state(Geom G, Layout L, int s, const double* __restrict__ u, const double* __restrict__ coef,
                             __nv_bfloat16* __restrict__ act) {
  const long long pts = (long long)G.Z * G.Y * G.X;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y), z = (int)(r / G.Y);
    const long long p = L.off0 + x + y * L.sy + z * L.sz;
    __align__(16) __nv_bfloat16 h[32];
#pragma unroll
    for (int c = 0; c < CH; ++c)
      h[c] = __float2bfloat16_rn(c < NV ? (float)((u[c * L.vs + p] - coef[c]) * coef[NV + c]) : 0.f);
    store_point(G, act, s, z, y, x, h);
  }
}

// Training target of sample s: (target_v - coarse_v) * out_scale_v / step_scale_v.
__global__ void k_pack_target(Geom G, Layout L, int s, const double* __restrict__ coarse,
                              const double* __restrict__ target, const double* __restrict__ coef,
                              float* __restrict__ t) {
  const long long pts = (long long)G.Z * G.Y * G.X;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y), z = (int)(r / G.Y);
    const long long p = L.off0 + x + y * L.sy + z * L.sz;
    float* o = t + ((long long)s * pts + i) * CH;
#pragma unroll
    for (int c = 0; c < CH; ++c)
      o[c] = c < NV ? (float)((target[c * L.vs + p] - coarse[c * L.vs + p]) * coef[2 * NV + c] / coef[3 * NV + c])
                    : 0.f;
  }
}

// One training pair packed into unpadded BF16 buffers: x = network input of
// the coarse state, t = normalised correction (target - coarse) * out_scale /
// step_scale (if target).
__global__ void k_pack_pair(Geom G, Layout L, const double* __restrict__ coarse, const double* __restrict__ target,
                            const double* __restrict__ coef, __nv_bfloat16* __restrict__ x,
                            __nv_bfloat16* __restrict__ t) {
  const long long pts = (long long)G.Z * G.Y * G.X;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int xx = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y), z = (int)(r / G.Y);
    const long long p = L.off0 + xx + y * L.sy + z * L.sz;
    __align__(16) __nv_bfloat16 hx[32], ht[32];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const double u = c < NV ? coarse[c * L.vs + p] : 0.0;
      hx[c] = __float2bfloat16_rn(c < NV ? (float)((u - coef[c]) * coef[NV + c]) : 0.f);
      if (target)
        ht[c] = __float2bfloat16_rn(
            c < NV ? (float)((target[c * L.vs + p] - u) * coef[2 * NV + c] / coef[3 * NV + c]) : 0.f);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) ((uint4*)(x + i * CH))[q] = ((const uint4*)hx)[q];
    if (target)
#pragma unroll
      for (int q = 0; q < 4; ++q) ((uint4*)(t + i * CH))[q] = ((const uint4*)ht)[q];
  }
}

__global__ void k_bf16_to_f32(long long n, const __nv_bfloat16* __restrict__ in, float* __restrict__ out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = __bfloat162float(in[i]);
}

// state += network output * step_scale / out_scale (interior, sample 0).
__global__ void k_apply(Geom G, Layout L, const float* __restrict__ out, const double* __restrict__ coef,
                        double* __restrict__ u) {
  const long long pts = (long long)G.Z * G.Y * G.X;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < pts; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % G.X);
    const long long r = i / G.X;
    const int y = (int)(r % G.Y), z = (int)(r / G.Y);
    const long long p = L.off0 + x + y * L.sy + z * L.sz;
#pragma unroll 4
    for (int c = 0; c < NV; ++c) u[c * L.vs + p] += (double)out[i * CH + c] * coef[3 * NV + c] / coef[2 * NV + c];
  }
}

// ---------------------------------------------------------------- MMA rate probe
// Back-to-back kind::f16 MMAs (M = 128, K = 16, N = NC) on no-swizzle
// operands in shared memory, one CTA per SM, issued the way the convolutions
// issue them: warp 0 runs the loop on warp-uniform descriptors whose A start
// moves by 0-2 entries from one MMA to the next (the taps' shifts) and one
// elected lane issues. The instruction-rate ceiling of those shapes.
constexpr int PROBE_A = 128 * 32, PROBE_B = 256 * 32, PROBE_SMEM = 1024 + PROBE_A + PROBE_B + 256;

template <int NC>
__global__ void __launch_bounds__(128, 1) k_mma_rate(int iters, unsigned long long* ns, unsigned int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bar = (uint64_t*)(base + PROBE_A + PROBE_B);
  uint32_t* slot = (uint32_t*)(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < (PROBE_A + PROBE_B) / 4; i += blockDim.x) ((uint32_t*)base)[i] = 0x3c003c00u;
  tc::fence_proxy_async();
  if (tid == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(slot, 256);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = *slot;
  if (warp == 0) {
    // A 128 x 16 and B NC x 16, K-major, core matrices 8 rows x 16 bytes
    const uint64_t ad = tc::smem_desc(tc::smem_u32(base), 2048, 128, tc::SWZ_NONE);
    const uint64_t bd = tc::smem_desc(tc::smem_u32(base + PROBE_A), NC * 16, 128, tc::SWZ_NONE);
    constexpr uint32_t IDESC = tc::idesc_bf16_f32(128, NC);
    const uint64_t t0 = tc::global_ns();
    for (int i = 0; i < iters; i += 6) {
#pragma unroll
      for (int t = 0; t < 6; ++t) tc::mma_bf16_elect(taddr, ad + (uint64_t)(t % 3), bd, IDESC, (i | t) ? 1u : 0u);
    }
    tc::mma_commit_elect(bar);
    const bool ok = tc::warp_wait(bar, 0);
    if (tid == 0) {
      ns[blockIdx.x] = tc::global_ns() - t0;
      if (!ok) atomicOr(err, 1u);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(taddr, 256);
}

// ---------------------------------------------------------------- failure-path probe
// The bounded waits and the abort handling of the warp-specialised tcgen05
// kernels, made to run out on purpose: warp 0 allocates TMEM; warp 1 issues
// one MMA (committed to `mma_done`), then waits with the caller's short limit
// on a barrier that nothing arrives at, gives up, records the timeout and
// raises the CTA abort flag, and waits (bounded) for its MMA before TMEM is
// released; warp 2 waits on a second such barrier with the kernels' default
// 2 s limit and is released by the abort flag instead. Warp 0 frees TMEM.
// done: bit 0 = TMEM freed, bit 1 = warp 2 left because of the abort.
__global__ void __launch_bounds__(96, 1) k_wait_timeout_probe(unsigned long long limit_ns, unsigned int* err,
                                                               unsigned int* done) {
  __shared__ __align__(1024) uint8_t ops[PROBE_A + 32 * 32];
  __shared__ uint64_t bars[3];  // 0 and 1: never arrived at; 2: MMA completion
  __shared__ uint32_t slot;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < (int)sizeof(ops) / 4; i += blockDim.x) ((uint32_t*)ops)[i] = 0u;
  tc::fence_proxy_async();
  if (tid == 0) {
    abort_flag = 0;
    for (int b = 0; b < 3; ++b) tc::mbar_init(&bars[b], 1);
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(&slot, 32);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = slot;
  if (warp == 1 && lane == 0) {
    const uint64_t ad = tc::smem_desc(tc::smem_u32(ops), 2048, 128, tc::SWZ_NONE);
    const uint64_t bd = tc::smem_desc(tc::smem_u32(ops + PROBE_A), 32 * 16, 128, tc::SWZ_NONE);
    tc::mma_bf16(taddr, ad, bd, tc::idesc_bf16_f32(128, 32), 0u);
    tc::mma_commit(&bars[2]);
    if (!tc::mbar_wait_or_abort(&bars[0], 0, &abort_flag, limit_ns)) {
      if (!abort_flag) atomicOr(err, 1u);
      abort_flag = 1;
    }
    tc::mbar_wait(&bars[2], 0);  // the MMA in flight lands before TMEM goes
  }
  if (warp == 2 && lane == 0) {
    if (!tc::mbar_wait_or_abort(&bars[1], 0, &abort_flag) && abort_flag) atomicOr(done, 2u);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(taddr, 32);
    if (lane == 0) atomicOr(done, 1u);
  }
}

// ---------------------------------------------------------------- host helpers
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

bool encode(CUtensorMap* tm, void* ptr, int rank, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
            const cuuint32_t* box, CUtensorMapSwizzle swz,
            CUtensorMapDataType type = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(tm, type, rank, ptr, dims, strides_bytes, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Padded chunk-major activations as a 5D tensor {8 channels, X+2, Y+2, 4
// chunks, S (Z+2) planes}, the first two as one where slab_rows; box {8, X+1,
// R+2, 4, 1} = one convolution slab
// (rows y0-1 .. y0+R of one plane, points x = 0 .. X including the zero pad
// at x = X), no swizzle: in shared memory [chunk][row][x][8 channels].
bool map_slab(CUtensorMap* tm, void* ptr, const Geom& G, int R) {
  const cuuint64_t row = 16ull * (G.X + 2), chunk = row * (G.Y + 2), planes = (cuuint64_t)G.S * (G.Z + 2);
  if (slab_rows(G.X)) {
    const cuuint64_t dims[4] = {2ull * (G.X + 2), (cuuint64_t)G.Y + 2, 4, planes};
    const cuuint64_t str[3] = {row, chunk, 4 * chunk};
    const cuuint32_t box[4] = {2 * (cuuint32_t)G.X + 2, (cuuint32_t)R + 2, 4, 1};
    return encode(tm, ptr, 4, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_DATA_TYPE_FLOAT64);
  }
  const cuuint64_t dims[5] = {8, (cuuint64_t)G.X + 2, (cuuint64_t)G.Y + 2, 4, planes};
  const cuuint64_t str[4] = {16, row, chunk, 4 * chunk};
  const cuuint32_t box[5] = {8, (cuuint32_t)G.X + 1, (cuuint32_t)R + 2, 4, 1};
  return encode(tm, ptr, 5, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

// weights [27*32 rows][32]: box {32, 32}, 64B swizzle
bool map_w(CUtensorMap* tm, void* ptr) {
  const cuuint64_t dims[2] = {CH, NTAP * CH};
  const cuuint64_t str[1] = {CH * 2};
  const cuuint32_t box[2] = {CH, CH};
  return encode(tm, ptr, 2, dims, str, box, CU_TENSOR_MAP_SWIZZLE_64B);
}

// Rows of the same activations for the weight gradient: {X+2 points of 16
// bytes as pairs of 8, Y+2, S (Z+2) planes, 4 chunks}, box {points, 1, 1, 4}:
// in shared memory [chunk][x][8 channels]. The points of a row are one
// dimension, so that a copy moves runs of 16 bytes times the points.
bool map_row(CUtensorMap* tm, void* ptr, const Geom& G, int points) {
  const cuuint64_t dims[4] = {2ull * (G.X + 2), (cuuint64_t)G.Y + 2, (cuuint64_t)G.S * (G.Z + 2), 4};
  const cuuint64_t row = 16ull * (G.X + 2), chunk = row * (G.Y + 2);
  const cuuint64_t str[3] = {row, 4 * chunk, chunk};
  const cuuint32_t box[4] = {2 * (cuuint32_t)points, 1, 1, 4};
  return encode(tm, ptr, 4, dims, str, box, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_DATA_TYPE_FLOAT64);
}

}  // namespace

// =========================================================================== corrector object
struct bssn_corrector {
  Geom G{};          // geometry at max batch
  int n = 0, max_batch = 0;
  long long pts = 0;        // max_batch * n^3
  long long pad_pts = 0;    // max_batch * (n+2)^3
  std::vector<void*> allocs;
  __nv_bfloat16* act[NL] = {};   // padded inputs of layers 1..5 (act[0] = network input)
  float* z[NL] = {};             // pre-activations (layer outputs), unpadded FP32
  __nv_bfloat16* g[2] = {};      // padded gradients (ping-pong)
  float* target = nullptr;       // unpadded FP32 targets
  float* partial = nullptr;      // wgrad partials
  double* lpart = nullptr;       // loss partials
  float* params = nullptr;       // FP32 master [NL][LAYER_PARAMS]
  float* grads = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  __nv_bfloat16* wf = nullptr;   // [NL][27][32][32]
  __nv_bfloat16* wb = nullptr;
  double* coef = nullptr;        // in_offset[24], in_scale[24], out_scale[24], step_scale[24]
  unsigned int* err = nullptr;
  int wg_blocks = 0, rows_per_cta = 0;
  int sms = 0;        // streaming multiprocessors (one conv CTA each)
  // convolution plans by sample count (the grid is fixed per network), so
  // that the search over (rows, planes) pairs runs once, not on every layer
  // launch
  ConvPlan plan[65];
  int plan_grid[65] = {};  // 0: not planned yet
  int conv_smem = 0;  // the most dynamic shared memory a convolution plan of this grid asks for
  long long adam_t = 0;
};

namespace {

cudaError_t calloc_dev(bssn_corrector* c, size_t bytes, void** p) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaSuccess) {
    c->allocs.push_back(*p);
    e = cudaMemset(*p, 0, bytes);
  }
  return e;
}

void corrector_free(bssn_corrector* c) {
  for (void* p : c->allocs) cudaFree(p);
  c->allocs.clear();
}

Geom geom_for(const bssn_corrector* c, int S) {
  Geom G = c->G;
  G.S = S;
  return G;
}

// Slab geometry for an X-wide grid and R output rows per unit: T 128-entry
// tiles cover the R (X+1) entries, K = 16 / T blocks of 32 TMEM columns per
// tile (512 columns), four slabs (128-byte aligned), the weights and the tail
// within the shared-memory limit. Returns false if it does not fit.
bool make_conv_plan(int X, int R, ConvPlan* out) {
  const int XS = X + 1;
  ConvPlan P{};
  P.R = R;
  P.T = (R * XS + 127) / 128;
  if (P.T > 8) return false;
  P.K = KMAX / P.T;
  P.chunk_bytes = (R + 2) * XS * 16;
  P.plane_bytes = 4 * P.chunk_bytes;
  P.slab_stride = (P.plane_bytes + 127) / 128 * 128;
  const int over = XS + 128 * P.T + XS + 1 - (R + 2) * XS;  // entries read past a slab (discarded rows)
  P.tail_bytes = over > 0 ? (over * 16 + 127) / 128 * 128 : 0;
  P.slab_off = NTAP * W_TAP_BYTES + 128;
  P.bar_off = P.slab_off + SLABS * P.slab_stride + P.tail_bytes;
  P.smem = std::max(1024 + P.bar_off + 512, CONV_SMEM_MIN);
  int cols = 32;
  while (cols < P.T * P.K * 32) cols *= 2;
  P.tmem_cols = cols;
  if (P.smem > CONV_SMEM_MAX) return false;
  *out = P;
  return true;
}

// The largest dynamic shared memory any row count of an X-wide, Y-high grid
// asks for (0 if none fits).
int conv_smem_max(int X, int Y) {
  int m = 0;
  for (int R = 1; R <= Y; ++R) {
    ConvPlan P;
    if (make_conv_plan(X, R, &P) && P.smem > m) m = P.smem;
  }
  return m;
}

// Work units for S samples: (sample, row block of R rows, run of L <= K
// planes). A unit issues T tiles x (L + 2) input planes of MMAs, so R and L
// are picked to make ceil(units / SMs) T (L + 2) smallest (then the fewest
// units). Returns the grid size, 0 if no plan fits.
int conv_units_search(const bssn_corrector* c, const Geom& G, ConvPlan* P) {
  double best = 1e300;
  long long best_units = 0;
  for (int R = 1; R <= G.Y; ++R) {
    ConvPlan Q;
    if (!make_conv_plan(G.X, R, &Q)) continue;
    Q.nyb = (G.Y + R - 1) / R;
    for (int L = 1; L <= Q.K && L <= G.Z; ++L) {
      const long long units = (long long)G.S * Q.nyb * ((G.Z + L - 1) / L);
      const long long slots = (long long)c->sms * CONV_CTAS;
      const double cost = (double)((units + slots - 1) / slots) * Q.T * (L + 2);
      if (cost < best || (cost == best && units < best_units)) {
        best = cost;
        best_units = units;
        *P = Q;
        P->L = L;
      }
    }
  }
  if (best == 1e300) return 0;
  P->nzs = (G.Z + P->L - 1) / P->L;
  const long long units = (long long)G.S * P->nyb * P->nzs;
  const long long slots = (long long)c->sms * CONV_CTAS;
  return (int)(units < slots ? units : slots);
}

int conv_units(bssn_corrector* c, const Geom& G, ConvPlan* P) {
  if (G.S < 1 || G.S > 64) return conv_units_search(c, G, P);
  if (!c->plan_grid[G.S]) c->plan_grid[G.S] = conv_units_search(c, G, &c->plan[G.S]);
  *P = c->plan[G.S];
  return c->plan_grid[G.S];
}

// one layer forward on act[l] (sample count in G) -> z[l] and act[l+1]
cudaError_t layer_forward(bssn_corrector* c, const Geom& G, int l, float* zout, __nv_bfloat16* act_out, int gelu,
                          cudaStream_t s) {
  ConvPlan P;
  const int grid = conv_units(c, G, &P);
  CUtensorMap ta, tw;
  if (grid < 1 || !map_slab(&ta, c->act[l], G, P.R) || !map_w(&tw, c->wf + (size_t)l * NTAP * CH * CH))
    return cudaErrorInvalidValue;
  const float* bias = c->params + (size_t)l * LAYER_PARAMS + NTAP * CH * CH;
  // programmatic dependent launch: the CTAs' set-up (barriers, TMEM, the
  // weights) overlaps the previous kernel's tail; the producer waits for the
  // previous kernel before it loads an activation slab
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(CONV_THREADS);
  cfg.dynamicSmemBytes = (size_t)P.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_conv_tc<0>, ta, tw, G, P, bias, zout, act_out, (const float*)nullptr, gelu,
                            c->err);
}

// the whole network; the last layer writes its output to `last` if given
// (the caller's buffer, same [S][n^3][32] layout), else to z[NL-1]. The
// hidden layers' pre-activations go to z[l] only with keep_pre (the backward
// pass reads them); inference writes just the activations.
cudaError_t network_forward(bssn_corrector* c, const Geom& G, cudaStream_t s, float* last = nullptr,
                            bool keep_pre = true) {
  cudaError_t e = cudaSuccess;
  for (int l = 0; l < NL && e == cudaSuccess; ++l) {
    float* zout = l == NL - 1 ? (last ? last : c->z[l]) : (keep_pre ? c->z[l] : nullptr);
    e = layer_forward(c, G, l, zout, l < NL - 1 ? c->act[l + 1] : nullptr, l < NL - 1 ? 1 : 0, s);
  }
  return e;
}

// backward through all layers given the output gradient in g[0] (padded BF16);
// fills c->grads.
cudaError_t network_backward(bssn_corrector* c, const Geom& G, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  int cur = 0;
  const long long rows = (long long)G.S * G.Z * G.Y;
  const int nb = c->wg_blocks;
  const int rpc = (int)((rows + nb - 1) / nb);
  for (int l = NL - 1; l >= 0 && e == cudaSuccess; --l) {
    float* gW = c->grads + (size_t)l * LAYER_PARAMS;
    CUtensorMap tx, tg;
    if (!map_row(&tx, c->act[l], G, G.X + 2) || !map_row(&tg, c->g[cur], G, G.X)) return cudaErrorInvalidValue;
    if (e == cudaSuccess) {
      if (G.X == 64)
        k_wgrad_rows<64><<<nb, WG_THREADS, WR<64>::SMEM, s>>>(tx, tg, G, rpc, c->partial, c->err);
      else
        k_wgrad_rows<32><<<nb, WG_THREADS, WR<32>::SMEM, s>>>(tx, tg, G, rpc, c->partial, c->err);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
      // weight and bias gradients (the bias follows the weights in gW)
      k_wgrad_reduce<<<(NTAP * CH * CH + CH + 31) / 32, 256, 0, s>>>(c->partial, nb, gW);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess && l > 0) {
      ConvPlan P;
      const int grid = conv_units(c, G, &P);
      CUtensorMap ta, tw;
      if (grid < 1 || !map_slab(&ta, c->g[cur], G, P.R) || !map_w(&tw, c->wb + (size_t)l * NTAP * CH * CH))
        return cudaErrorInvalidValue;
      k_conv_tc<1><<<grid, CONV_THREADS, P.smem, s>>>(ta, tw, G, P, nullptr, nullptr, c->g[1 - cur], c->z[l - 1], 0,
                                                      c->err);
      e = cudaGetLastError();
      cur = 1 - cur;
    }
  }
  return e;
}

cudaError_t refresh_weights(bssn_corrector* c, cudaStream_t s) {
  k_weights_bf16<<<dim3((NTAP * CH * CH + 255) / 256, NL), 256, 0, s>>>(c->params, c->wf, c->wb);
  return cudaGetLastError();
}

// loss and output gradient for targets in c->target, or for the samples' BF16
// ones if given; returns the loss (synchronizes)
cudaError_t loss_and_grad(bssn_corrector* c, const Geom& G, double* loss, cudaStream_t s,
                          const TargetsBf16* bf16 = nullptr) {
  if (bf16)
    k_mse<<<MSE_BLOCKS, MSE_THREADS, 0, s>>>(G, NV, c->z[NL - 1], *bf16, c->g[0], c->lpart);
  else
    k_mse<<<MSE_BLOCKS, MSE_THREADS, 0, s>>>(G, NV, c->z[NL - 1], TargetsF32{c->target}, c->g[0], c->lpart);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = network_backward(c, G, s);
  double h[MSE_BLOCKS];
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, c->lpart, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess) {
    double sum = 0.0;
    for (int i = 0; i < MSE_BLOCKS; ++i) sum += h[i];
    *loss = sum / ((double)G.S * G.Z * G.Y * G.X * NV);
  }
  return e;
}

bssn_status_t status_of(bssn_corrector* c, cudaError_t e, cudaStream_t s) {
  if (e != cudaSuccess) return e == cudaErrorInvalidValue ? BSSN_ERR_UNSUPPORTED : BSSN_ERR_CUDA;
  unsigned int err = 0;
  e = cudaMemcpyAsync(&err, c->err, sizeof(err), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return BSSN_ERR_CUDA;
  return err ? BSSN_ERR_TIMEOUT : BSSN_OK;
}

}  // namespace

extern "C" {

bssn_status_t bssn_corrector_create(bssn_corrector_t** out, int n, int max_batch, unsigned long long seed) {
  if (!out || (n != 32 && n != 64 && n != 128) || max_batch < 1 || max_batch > 64) return BSSN_ERR_INVALID_ARG;
  *out = nullptr;
  if (!encode_fn()) return BSSN_ERR_UNSUPPORTED;
  bssn_corrector* c = new (std::nothrow) bssn_corrector;
  if (!c) return BSSN_ERR_NOMEM;
  c->n = n;
  c->max_batch = max_batch;
  c->G = Geom{max_batch, n, n, n};
  c->pts = (long long)max_batch * n * n * n;
  c->pad_pts = (long long)max_batch * (n + 2) * (n + 2) * (n + 2);
  // one weight-gradient CTA per SM (each streams a range of rows)
  {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || sms < 1)
      sms = 128;
    const long long rows = (long long)max_batch * n * n;
    c->wg_blocks = (int)(rows < sms ? rows : sms);
  }
  cudaError_t e = cudaSuccess;
  void* p = nullptr;
  for (int l = 0; l < NL && e == cudaSuccess; ++l) {
    e = calloc_dev(c, c->pad_pts * CH * 2, &p);
    c->act[l] = (__nv_bfloat16*)p;
    if (e == cudaSuccess) e = calloc_dev(c, c->pts * CH * 4, &p);
    c->z[l] = (float*)p;
  }
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
    e = calloc_dev(c, c->pad_pts * CH * 2, &p);
    c->g[i] = (__nv_bfloat16*)p;
  }
  if (e == cudaSuccess) e = calloc_dev(c, c->pts * CH * 4, &p);
  c->target = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, (size_t)c->wg_blocks * (NTAP * CH * CH + CH) * 4, &p);
  c->partial = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, MSE_BLOCKS * sizeof(double), &p);
  c->lpart = (double*)p;
  const size_t np = (size_t)NL * LAYER_PARAMS;
  if (e == cudaSuccess) e = calloc_dev(c, np * 4, &p);
  c->params = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, np * 4, &p);
  c->grads = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, np * 4, &p);
  c->adam_m = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, np * 4, &p);
  c->adam_v = (float*)p;
  if (e == cudaSuccess) e = calloc_dev(c, (size_t)NL * NTAP * CH * CH * 2, &p);
  c->wf = (__nv_bfloat16*)p;
  if (e == cudaSuccess) e = calloc_dev(c, (size_t)NL * NTAP * CH * CH * 2, &p);
  c->wb = (__nv_bfloat16*)p;
  if (e == cudaSuccess) e = calloc_dev(c, 4 * NV * sizeof(double), &p);
  c->coef = (double*)p;
  if (e == cudaSuccess) e = calloc_dev(c, sizeof(unsigned int), &p);
  c->err = (unsigned int*)p;
  c->conv_smem = conv_smem_max(n, n);
  if (e == cudaSuccess && c->conv_smem == 0) e = cudaErrorInvalidValue;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv_tc<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, c->conv_smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, c->conv_smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad_rows<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, WR<64>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad_rows<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, WR<32>::SMEM);
  // ask for the full shared-memory carveout for the tensor-core kernels
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv_tc<0>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_conv_tc<1>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad_rows<64>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad_rows<32>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess) {
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev);
  }
  // seeded initialisation: uniform in +-sqrt(6 / fan_in) (real fan-in), the
  // last layer scaled by 0.1 so the initial correction is small; biases 0;
  // weights of padded channels 0
  if (e == cudaSuccess) {
    std::vector<float> h(np, 0.f);
    uint64_t st = seed ^ 0x5DEECE66DULL;
    auto next = [&]() {
      st += 0x9E3779B97F4A7C15ULL;
      uint64_t zz = st;
      zz = (zz ^ (zz >> 30)) * 0xBF58476D1CE4E5B9ULL;
      zz = (zz ^ (zz >> 27)) * 0x94D049BB133111EBULL;
      zz ^= zz >> 31;
      return (double)(zz >> 11) * (1.0 / 9007199254740992.0);
    };
    const int cin[NL] = {NV, CH, CH, CH, CH}, cout[NL] = {CH, CH, CH, CH, NV};
    for (int l = 0; l < NL; ++l) {
      const double bound = std::sqrt(6.0 / (27.0 * cin[l])) * (l == NL - 1 ? 0.1 : 1.0);
      for (int t = 0; t < NTAP; ++t)
        for (int co = 0; co < CH; ++co)
          for (int ci = 0; ci < CH; ++ci) {
            const double r = next();
            if (co < cout[l] && ci < cin[l])
              h[(size_t)l * LAYER_PARAMS + ((size_t)t * CH + co) * CH + ci] = (float)((2 * r - 1) * bound);
          }
    }
    e = cudaMemcpy(c->params, h.data(), np * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = refresh_weights(c, 0);
    std::vector<double> cf(4 * NV, 1.0);
    for (int v = 0; v < NV; ++v) cf[v] = 0.0;
    if (e == cudaSuccess) e = cudaMemcpy(c->coef, cf.data(), 4 * NV * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    corrector_free(c);
    delete c;
    return e == cudaErrorMemoryAllocation ? BSSN_ERR_NOMEM : BSSN_ERR_CUDA;
  }
  *out = c;
  return BSSN_OK;
}

bssn_status_t bssn_corrector_destroy(bssn_corrector_t* c) {
  if (!c) return BSSN_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  corrector_free(c);
  delete c;
  return BSSN_OK;
}

long long bssn_corrector_param_count(void) { return (long long)NL * LAYER_PARAMS; }

bssn_status_t bssn_corrector_layer_output(bssn_corrector_t* c, int layer, int S, float* out) {
  if (!c || !out || layer < 0 || layer >= NL || S < 1 || S > c->max_batch) return BSSN_ERR_INVALID_ARG;
  return cudaMemcpy(out, c->z[layer], (size_t)S * c->n * c->n * c->n * CH * 4, cudaMemcpyDeviceToDevice) ==
                 cudaSuccess
             ? BSSN_OK
             : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_params(bssn_corrector_t* c, float* host, int write) {
  if (!c || !host) return BSSN_ERR_INVALID_ARG;
  const size_t bytes = (size_t)NL * LAYER_PARAMS * 4;
  cudaError_t e;
  if (write) {
    e = cudaMemcpy(c->params, host, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = refresh_weights(c, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  } else {
    e = cudaMemcpy(host, c->params, bytes, cudaMemcpyDeviceToHost);
  }
  return e == cudaSuccess ? BSSN_OK : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_grads(bssn_corrector_t* c, float* host) {
  if (!c || !host) return BSSN_ERR_INVALID_ARG;
  return cudaMemcpy(host, c->grads, (size_t)NL * LAYER_PARAMS * 4, cudaMemcpyDeviceToHost) == cudaSuccess
             ? BSSN_OK
             : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_set_scales(bssn_corrector_t* c, const double* in_offset, const double* in_scale,
                                        const double* out_scale) {
  if (!c || !in_offset || !in_scale || !out_scale) return BSSN_ERR_INVALID_ARG;
  double h[3 * NV];
  for (int v = 0; v < NV; ++v) {
    if (!std::isfinite(in_offset[v]) || !(in_scale[v] > 0) || !(out_scale[v] > 0)) return BSSN_ERR_INVALID_ARG;
    h[v] = in_offset[v];
    h[NV + v] = in_scale[v];
    h[2 * NV + v] = out_scale[v];
  }
  return cudaMemcpy(c->coef, h, sizeof(h), cudaMemcpyHostToDevice) == cudaSuccess ? BSSN_OK : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_set_step_scale(bssn_corrector_t* c, const double* step_scale) {
  if (!c || !step_scale) return BSSN_ERR_INVALID_ARG;
  for (int v = 0; v < NV; ++v)
    if (!(step_scale[v] > 0) || !std::isfinite(step_scale[v])) return BSSN_ERR_INVALID_ARG;
  return cudaMemcpy(c->coef + 3 * NV, step_scale, NV * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess
             ? BSSN_OK
             : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_forward_raw(bssn_corrector_t* c, int S, const void* x_bf16, float* out, void* stream) {
  if (!c || !x_bf16 || !out || S < 1 || S > c->max_batch) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, S);
  cudaError_t e = cudaMemsetAsync(c->err, 0, 4, s);
  if (e == cudaSuccess) {
    k_pad_copy<<<1024, 256, 0, s>>>(G, (const __nv_bfloat16*)x_bf16, c->act[0]);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = network_forward(c, G, s, out);
  return status_of(c, e, s);
}

bssn_status_t bssn_corrector_infer_async(bssn_corrector_t* c, int S, const void* x_bf16, float* out, void* stream) {
  if (!c || !x_bf16 || !out || S < 1 || S > c->max_batch) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, S);
  k_pad_copy<<<1024, 256, 0, s>>>(G, (const __nv_bfloat16*)x_bf16, c->act[0]);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = network_forward(c, G, s, out, false);
  if (e != cudaSuccess) return e == cudaErrorInvalidValue ? BSSN_ERR_UNSUPPORTED : BSSN_ERR_CUDA;
  return BSSN_OK;
}

bssn_status_t bssn_corrector_sync(bssn_corrector_t* c, void* stream) {
  if (!c) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, c->err, sizeof(err), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->err, 0, sizeof(err), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return BSSN_ERR_CUDA;
  return err ? BSSN_ERR_TIMEOUT : BSSN_OK;
}

bssn_status_t bssn_corrector_loss_grad_raw(bssn_corrector_t* c, int S, const void* x_bf16, const float* target,
                                           double* loss, void* stream) {
  if (!c || !x_bf16 || !target || !loss || S < 1 || S > c->max_batch) return BSSN_ERR_INVALID_ARG;
  if (c->n > 64) return BSSN_ERR_UNSUPPORTED;  // the weight gradient walks whole x-rows of 32 or 64 points
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, S);
  cudaError_t e = cudaMemsetAsync(c->err, 0, 4, s);
  if (e == cudaSuccess) {
    k_pad_copy<<<1024, 256, 0, s>>>(G, (const __nv_bfloat16*)x_bf16, c->act[0]);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(c->target, target, (size_t)S * c->n * c->n * c->n * CH * 4, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = network_forward(c, G, s);
  if (e == cudaSuccess) e = loss_and_grad(c, G, loss, s);
  return status_of(c, e, s);
}

bssn_status_t bssn_corrector_train_step(bssn_corrector_t* c, const bssn_grid_t* grid, int S,
                                        const double* const* coarse, const double* const* target, float lr,
                                        double* loss, void* stream) {
  if (!c || !grid || !coarse || !target || !loss || S < 1 || S > c->max_batch) return BSSN_ERR_INVALID_ARG;
  if (c->n > 64) return BSSN_ERR_UNSUPPORTED;  // the weight gradient walks whole x-rows of 32 or 64 points
  if (grid->nx != c->n || grid->ny != c->n || grid->nz != c->n || !(lr >= 0)) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, S);
  const Layout L = make_layout(*grid);
  cudaError_t e = cudaMemsetAsync(c->err, 0, 4, s);
  for (int i = 0; i < S && e == cudaSuccess; ++i) {
    if (!coarse[i] || !target[i]) return BSSN_ERR_INVALID_ARG;
    k_pack_state<<<512, 256, 0, s>>>(G, L, i, coarse[i], c->coef, c->act[0]);
    k_pack_target<<<512, 256, 0, s>>>(G, L, i, coarse[i], target[i], c->coef, c->target);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = network_forward(c, G, s);
  if (e == cudaSuccess) e = loss_and_grad(c, G, loss, s);
  if (e == cudaSuccess && lr > 0) {
    c->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)c->adam_t), c2 = 1.f - powf(b2, (float)c->adam_t);
    const int np = NL * LAYER_PARAMS;
    k_adam<<<(np + 255) / 256, 256, 0, s>>>(np, c->params, c->grads, c->adam_m, c->adam_v, lr, b1, b2, 1e-8f, c1, c2);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = refresh_weights(c, s);
  }
  return status_of(c, e, s);
}

bssn_status_t bssn_corrector_pack(bssn_corrector_t* c, const bssn_grid_t* grid, const double* coarse,
                                  const double* target, void* x_bf16, void* t_bf16, void* stream) {
  if (!c || !grid || !coarse || !x_bf16 || (target && !t_bf16)) return BSSN_ERR_INVALID_ARG;
  if (grid->nx != c->n || grid->ny != c->n || grid->nz != c->n) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  k_pack_pair<<<512, 256, 0, s>>>(geom_for(c, 1), make_layout(*grid), coarse, target, c->coef,
                                  (__nv_bfloat16*)x_bf16, (__nv_bfloat16*)t_bf16);
  return cudaGetLastError() == cudaSuccess ? BSSN_OK : BSSN_ERR_CUDA;
}

bssn_status_t bssn_corrector_train_step_raw(bssn_corrector_t* c, int S, const void* const* x_bf16,
                                            const void* const* t_bf16, float lr, double* loss, void* stream) {
  if (!c || !x_bf16 || !t_bf16 || !loss || S < 1 || S > c->max_batch || !(lr >= 0)) return BSSN_ERR_INVALID_ARG;
  if (c->n > 64) return BSSN_ERR_UNSUPPORTED;  // the weight gradient walks whole x-rows of 32 or 64 points
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, S);
  const Geom G1 = geom_for(c, 1);
  const long long pts1 = (long long)c->n * c->n * c->n;
  const long long pad1 = (long long)(c->n + 2) * (c->n + 2) * (c->n + 2);
  // targets on 16-byte boundaries are read by the loss itself; others are
  // widened to FP32 first (14 us more per sample of 64^3)
  TargetsBf16 bf16{};
  bool wide = true;
  for (int i = 0; i < S; ++i) wide = wide && ((uintptr_t)t_bf16[i] & 15) == 0;
  cudaError_t e = cudaMemsetAsync(c->err, 0, 4, s);
  for (int i = 0; i < S && e == cudaSuccess; ++i) {
    if (!x_bf16[i] || !t_bf16[i]) return BSSN_ERR_INVALID_ARG;
    k_pad_copy<<<512, 256, 0, s>>>(G1, (const __nv_bfloat16*)x_bf16[i], c->act[0] + i * pad1 * CH);
    bf16.p[i] = (const __nv_bfloat16*)t_bf16[i];
    if (!wide) k_bf16_to_f32<<<512, 256, 0, s>>>(pts1 * CH, bf16.p[i], c->target + i * pts1 * CH);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = network_forward(c, G, s);
  if (e == cudaSuccess) e = loss_and_grad(c, G, loss, s, wide ? &bf16 : nullptr);
  if (e == cudaSuccess && lr > 0) {
    c->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)c->adam_t), c2 = 1.f - powf(b2, (float)c->adam_t);
    const int np = NL * LAYER_PARAMS;
    k_adam<<<(np + 255) / 256, 256, 0, s>>>(np, c->params, c->grads, c->adam_m, c->adam_v, lr, b1, b2, 1e-8f, c1, c2);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = refresh_weights(c, s);
  }
  return status_of(c, e, s);
}

bssn_status_t bssn_corrector_apply(bssn_corrector_t* c, const bssn_grid_t* grid, double* state, void* stream) {
  if (!c || !grid || !state) return BSSN_ERR_INVALID_ARG;
  if (grid->nx != c->n || grid->ny != c->n || grid->nz != c->n) return BSSN_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const Geom G = geom_for(c, 1);
  const Layout L = make_layout(*grid);
  cudaError_t e = cudaMemsetAsync(c->err, 0, 4, s);
  if (e == cudaSuccess) {
    k_pack_state<<<512, 256, 0, s>>>(G, L, 0, state, c->coef, c->act[0]);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = network_forward(c, G, s, nullptr, false);
  if (e == cudaSuccess) {
    k_apply<<<512, 256, 0, s>>>(G, L, c->z[NL - 1], c->coef, state);
    e = cudaGetLastError();
  }
  return status_of(c, e, s);
}

// Runs the failure-path probe once (one CTA) and reports what it did.
bssn_status_t bssn_probe_wait_timeout(unsigned long long limit_ns, unsigned int* flags) {
  if (!flags || limit_ns < 1000ull || limit_ns > 1000000000ull) return BSSN_ERR_INVALID_ARG;
  unsigned int* words = nullptr;
  cudaError_t e = cudaMalloc(&words, 2 * sizeof(unsigned int));
  if (e == cudaSuccess) e = cudaMemset(words, 0, 2 * sizeof(unsigned int));
  if (e == cudaSuccess) {
    k_wait_timeout_probe<<<1, 96>>>(limit_ns, words, words + 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  unsigned int h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpy(h, words, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(words);
  if (e != cudaSuccess) return BSSN_ERR_CUDA;
  *flags = h[1];
  return h[0] ? BSSN_ERR_TIMEOUT : BSSN_OK;
}

// Measured dense BF16 rate (TFLOP/s, all SMs) of back-to-back M=128 K=16
// tcgen05 MMAs with N = n (32, 64, 128 or 256) columns.
bssn_status_t bssn_probe_mma_rate(int n, double* tflops) {
  if (!tflops || (n != 32 && n != 64 && n != 96 && n != 128 && n != 256)) return BSSN_ERR_INVALID_ARG;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return BSSN_ERR_CUDA;
  void (*kern)(int, unsigned long long*, unsigned int*) =
      n == 32    ? k_mma_rate<32>
      : n == 64  ? k_mma_rate<64>
      : n == 96  ? k_mma_rate<96>
      : n == 128 ? k_mma_rate<128>
                 : k_mma_rate<256>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PROBE_SMEM);
  unsigned long long* ns = nullptr;
  unsigned int* err = nullptr;
  if (e == cudaSuccess) e = cudaMalloc(&ns, sizeof(unsigned long long) * sms);
  if (e == cudaSuccess) e = cudaMalloc(&err, sizeof(unsigned int));
  if (e == cudaSuccess) e = cudaMemset(err, 0, sizeof(unsigned int));
  const int iters = 4098;  // a multiple of 6
  std::vector<unsigned long long> h(sms);
  unsigned int herr = 0;
  for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {  // the first launch warms up
    kern<<<sms, 128, PROBE_SMEM>>>(iters, ns, err);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (e == cudaSuccess) e = cudaMemcpy(h.data(), ns, sizeof(unsigned long long) * sms, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(&herr, err, sizeof(unsigned int), cudaMemcpyDeviceToHost);
  cudaFree(ns);
  cudaFree(err);
  if (e != cudaSuccess) return BSSN_ERR_CUDA;
  if (herr) return BSSN_ERR_TIMEOUT;
  unsigned long long mx = 1;
  for (unsigned long long v : h) mx = v > mx ? v : mx;
  *tflops = 2.0 * 128.0 * n * 16.0 * iters * sms / (mx * 1e-9) / 1e12;
  return BSSN_OK;
}

}  // extern "C"
