// lbm_tile.cu -- the FP32 step of small and narrow domains: one tile per CTA.
//
// The ring kernel (lbm_fused.cu) is made for states that stream from HBM: a
// CTA sweeps many rows behind a TMA ring.  On a domain of a few rows per CTA
// its step is a chain of latencies instead (tensor-map fetch, TMA, three rows
// through one barrier each, two ghost rows): 5.5 us at 256 x 128, where the
// bytes need 0.35 us.  Here every node of a 64-column x R-row tile has its own
// thread (two nodes per thread, one warp per row), so a step is one plain load
// of the nine populations, rho and psi into shared memory, one barrier (two in
// the tiles at a wall), the collision and the stores; between kernels a CUDA
// graph needs 1.3 us.  The rows above and below the tile are loaded twice (from
// L2, which holds small states): with R = 4 half of the loads are repeats, with
// R = 6 a third.  56 registers (the launch bounds hold them there), against the
// ring kernel's 128, let an SM hold 35 warps.  The smallest domains make two
// steps per launch (k_pair).  The arithmetic is that of the ring kernel, bit for
// bit (lbm_node.cuh).
//
// Measured, us per step, Carnahan-Starling with general rates, ring -> tile:
// 64 x 32 3.9 -> 2.0, 256 x 128 5.5 -> 2.3, 400 x 200 5.9 -> 3.1, 512 x 512
// 7.9 -> 5.4, 1024 x 512 11.4 -> 8.5, 1024 x 1024 17.3 -> 15.1.
#include <stdlib.h>

#include "lbm_fused.h"
#include "lbm_tile.cuh"

namespace {

using lbm_tile::kW;

struct TileArgs : lbm_fused_args {
  static constexpr bool short_math = true;
};

template <bool UNIT, int MCW, int KIND, int R>
__global__ void __launch_bounds__((R + 3) * 32, R == 4 ? 5 : 4) k_tile(const float *__restrict__ fin, TileArgs P) {
  __shared__ lbm_tile::Smem<R> M;
  if (P.pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  lbm_tile::step<UNIT, MCW, KIND, R>(
      P, (int)blockIdx.x * kW, P.y0 + (int)blockIdx.y * R, fin, P.fout, M,
      [&] {
        // a direct launch is a programmatic dependent of the step before it: from
        // here on its stores are visible
        if (P.pdl) asm volatile("griddepcontrol.wait;" ::: "memory");
      },
      [&] {
        if (*(volatile int *)P.flag == 0) atomicOr(P.flag, 1);
      });
}

// Two steps per launch (tiles of kPairW columns x 4 rows).
constexpr int kPairR = 8;

template <bool UNIT, int MCW, int KIND>
__global__ void __launch_bounds__((kPairR + 3) * 32) k_pair(const float *__restrict__ fin, TileArgs P) {
  __shared__ lbm_tile::PairSmem<kPairR> S;
  if (P.pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  lbm_tile::step_pair<UNIT, MCW, KIND, kPairR>(
      P, (int)blockIdx.x * lbm_tile::kPairW, P.y0 + (int)blockIdx.y * (kPairR - 4), fin, P.fout, S,
      [&] {
        if (P.pdl) asm volatile("griddepcontrol.wait;" ::: "memory");
      },
      [&] {
        if (*(volatile int *)P.flag == 0) atomicOr(P.flag, 1);
      });
}

typedef void (*TileKernel)(const float *, TileArgs);
template <bool UNIT, int MCW, int KIND>
TileKernel pick(int rows) {  // rows of a tile; 0: two steps
  return rows == 4 ? (TileKernel)k_tile<UNIT, MCW, KIND, 4>
                   : (rows == 6 ? (TileKernel)k_tile<UNIT, MCW, KIND, 6> : (TileKernel)k_pair<UNIT, MCW, KIND>);
}
template <bool UNIT, int MCW>
TileKernel pick(int kind, int rows) {
  return kind == LBM_EOS_CARNAHAN_STARLING ? pick<UNIT, MCW, LBM_EOS_CARNAHAN_STARLING>(rows)
                                           : pick<UNIT, MCW, LBM_EOS_PIECEWISE>(rows);
}
TileKernel kernel_ptr(const lbm_ctx *C, int rows) {
  const int kind = C->dp.eos_kind;
  if (C->dp.wetting == LBM_WET_MARTYS_CHEN) return C->fused_unit ? pick<true, 1>(kind, rows) : pick<false, 1>(kind, rows);
  return C->fused_unit ? pick<true, 0>(kind, rows) : pick<false, 0>(kind, rows);
}

}  // namespace

// Which kernel runs a domain, by the columns x rows each works through (the ring's
// strips of 256 columns, the tile's of 64), from measurements of both.  While the
// two state arrays (72 bytes per node) mostly stay in the 126 MB L2 the tile kernel
// wins, past it the ring's deep prefetch does; the ring waits ~1.4 us for the ghost
// rows of a walled domain.  us per step, ring / tile (6 rows), unit | general rates:
//    walled    1280 x 1100 22.4 / 21.1 | 22.6 / 21.7, 1280 x 1200 23.4 / 24.2 | 23.5 / 24.4,
//              1792 x 960 26.8 / 27.3 | 27.1 / 27.8, 2048 x 960 29.3 / 30.8 | 29.6 / 31.5,
//              4096 x 2048 103 / 118 | 107 / 120;
//    periodic  1024 x 1300 19.7 / 19.3 | 20.5 / 20.0, 1536 x 900 20.0 / 20.4 | 20.7 / 21.1.
// Beyond, the tile wins where the ring's strips hold a tenth more columns than the
// domain (threads past nx idle): walled 448 x 3600 26.2 / 25.2 | 27.6 / 25.7,
// 1344 x 1344 30.1 / 28.5 | 29.8 / 29.6, 2624 x 1500 55.8 / 58.3 | 55.5 / 59.2,
// 320 x 8000 53 / 39 | 56 / 40.
// Tiles of 4 rows up to a million nodes (more CTAs, a shorter CTA: 400 x 200 3.08
// against 3.30 us, 1000 x 800 11.7 / 12.0, 1024 x 960 13.6 / 13.7), of 6 rows above
// (fewer repeated loads: 1024 x 1024 14.6 against 14.5, 1280 x 1000 19.4 / 18.4).
// Two steps per launch up to 50,000 nodes, where the launch and the loads are
// most of a step and two thirds of the collisions can be made twice, as long as the
// CTAs fit on the chip at once: us per step, one / two, 64 x 32 2.43 / 1.96, 256 x 128
// 2.50 / 2.22, 300 x 150 2.75 / 2.34; still 256 x 200 2.79 / 2.18 and 348 x 200
// 2.76 / 2.22, which the line leaves out, then 400 x 200 3.08 / 3.51; the other way
// round for tall and narrow domains below it, 60 x 800 2.63 / 3.09.
// The ring kernel's own tuning variables ask for the ring.
void lbm_tile_plan(lbm_ctx *C) {
  C->tile_rows = C->tile_pairs = 0;
  if (getenv("LBM_FUSED_STAGES") || getenv("LBM_FUSED_CTAS_PER_SM")) return;
  const long long nodes = (long long)C->nx * C->ny;
  const int strips = (C->nx + kW - 1) / kW, ring_cols = (C->nx + 255) / 256 * 256;
  const int nrows = C->walls ? C->ny - 2 : C->ny;
  if (1LL * strips * kW * C->ny > (C->walls ? 1420000 : 1360000) && 100LL * strips * kW > 90LL * ring_cols) return;
  const int R = nodes <= 1000000 ? 4 : 6, bands = (nrows + R - 1) / R;
  if (bands > 65535) return;  // grid.y
  C->tile_rows = R;
  C->tile_pairs = nodes <= 50000 && C->nx >= 8;
  C->tile_w = kW;
  C->tile_stages = 0;
  C->tile_blocks = strips * bands;
}

namespace {

// grid of tiles of w columns x r rows
cudaError_t launch(const lbm_ctx *C, int rows, int w, int r, int threads, const void *src, void *dst,
                   unsigned long long *launches) {
  TileArgs P{lbm_make_fused_args(C)};
  P.fout = (float *)dst;
  P.pdl = !C->capturing;
  // One after the other on a stream, plain launches of a short kernel are 4.1 us
  // apart and programmatically dependent ones 1.5 us; captured ones 1.3 us with
  // plain graph edges, which they keep (400 x 200 step without graphs: 6.2 ->
  // 3.75 us).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((C->nx + w - 1) / w, (P.nrows + r - 1) / r);
  cfg.blockDim = dim3(threads);
  cfg.stream = C->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = P.pdl;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel_ptr(C, rows), (const float *)src, P);
  ++*launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t lbm_tile_step(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches) {
  return launch(C, C->tile_rows, kW, C->tile_rows, (C->tile_rows + 3) * 32, src, dst, launches);
}

cudaError_t lbm_tile_pair(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches) {
  return launch(C, 0, lbm_tile::kPairW, kPairR - 4, (kPairR + 3) * 32, src, dst, launches);
}
