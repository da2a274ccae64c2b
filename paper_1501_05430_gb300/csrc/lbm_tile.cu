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
// 64 x 32 3.9 -> 1.9, 256 x 128 5.5 -> 2.3, 400 x 200 5.9 -> 3.1, 512 x 512
// 7.9 -> 5.6, 1024 x 512 11.4 -> 8.5, 1024 x 1024 17.3 -> 15.0.
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

// Which kernel runs a domain, from measurements of both (us per step, general
// rates, ring / tile of 6 rows):
//  - while both state arrays (72 bytes per node) stay in the 126 MB L2 the tile
//    kernel wins: 1280 x 1280 28.5 / 26.8, 1400 x 1200 28.4 / 27.4; past it the
//    ring's deep prefetch does: 2048 x 1024 31.3 / 33.2, 4096 x 2048 107 / 119;
//  - at any size where the ring's 256-column strips hold over a ninth more
//    columns than the tile's 64-column ones (its threads past nx idle):
//    128 x 32000 98.8 / 59.1, 300 x 8000 56.7 / 39.5, 640 x 8000 82.4 / 76.5,
//    1344 x 2048 44.5 / 43.2; at 720 x 6000, equal columns, 64.8 / 67.5.
// Tiles of 4 rows up to 2^20 nodes (more CTAs, a shorter CTA: 256 x 128 2.95
// against 3.26 us, 1024 x 512 9.1 / 9.4), of 6 rows above (fewer repeated
// loads: 1200 x 1200 23.9 against 22.9).
// Two steps per launch up to 50,000 nodes, where the launch and the loads are
// most of a step and two thirds of the collisions can be made twice: us per step,
// one / two, 64 x 32 2.65 / 2.07, 256 x 128 2.92 / 2.49, 300 x 100 2.91 / 2.20;
// 400 x 200 3.52 / 3.91.
// The ring kernel's own tuning variables ask for the ring.
void lbm_tile_plan(lbm_ctx *C) {
  C->tile_rows = C->tile_pairs = 0;
  if (getenv("LBM_FUSED_STAGES") || getenv("LBM_FUSED_CTAS_PER_SM")) return;
  const long long nodes = (long long)C->nx * C->ny;
  const int strips = (C->nx + kW - 1) / kW, ring_cols = (C->nx + 255) / 256 * 256;
  const int nrows = C->walls ? C->ny - 2 : C->ny;
  if (nodes > 1600000 && 10LL * strips * kW > 9LL * ring_cols) return;
  const int R = nodes <= (1 << 20) ? 4 : 6, bands = (nrows + R - 1) / R;
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
