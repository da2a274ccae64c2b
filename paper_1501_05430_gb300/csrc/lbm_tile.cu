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
// graph needs 1.3 us, the lower limit of a step.  The rows above and below the
// tile are loaded twice (from L2, which holds small states): with R = 4 half
// of the loads are repeats, with R = 6 a third.  56-60 registers, against the
// ring kernel's 128, let an SM hold 32 warps.  The arithmetic is that of the
// ring kernel, bit for bit (lbm_node.cuh).
//
// Measured, us per step, Carnahan-Starling with general rates, ring -> tile:
// 64 x 32 3.9 -> 2.8, 256 x 128 5.5 -> 2.9, 400 x 200 5.9 -> 3.6, 512 x 512
// 7.9 -> 5.8, 1024 x 512 11.4 -> 9.1, 1024 x 1024 17.3 -> 15.8.
#include <stdlib.h>

#include "lbm_fused.h"
#include "lbm_tile.cuh"

namespace {

using lbm_tile::kW;

template <bool UNIT, int MCW, int KIND, int R>
__global__ void __launch_bounds__((R + 3) * 32) k_tile(const float *__restrict__ fin, lbm_fused_args P) {
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

typedef void (*TileKernel)(const float *, lbm_fused_args);
template <bool UNIT, int MCW, int R>
TileKernel pick_kind(int kind) {
  return kind == LBM_EOS_CARNAHAN_STARLING ? (TileKernel)k_tile<UNIT, MCW, LBM_EOS_CARNAHAN_STARLING, R>
                                           : (TileKernel)k_tile<UNIT, MCW, LBM_EOS_PIECEWISE, R>;
}
template <int R>
TileKernel pick(bool unit, bool mc, int kind) {
  if (mc) return unit ? pick_kind<true, 1, R>(kind) : pick_kind<false, 1, R>(kind);
  return unit ? pick_kind<true, 0, R>(kind) : pick_kind<false, 0, R>(kind);
}
TileKernel kernel_ptr(const lbm_ctx *C) {
  const bool mc = C->dp.wetting == LBM_WET_MARTYS_CHEN;
  return C->tile_rows == 4 ? pick<4>(C->fused_unit, mc, C->dp.eos_kind) : pick<6>(C->fused_unit, mc, C->dp.eos_kind);
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
// The ring kernel's own tuning variables ask for the ring.
void lbm_tile_plan(lbm_ctx *C) {
  C->tile_rows = 0;
  if (getenv("LBM_FUSED_STAGES") || getenv("LBM_FUSED_CTAS_PER_SM")) return;
  const long long nodes = (long long)C->nx * C->ny;
  const int strips = (C->nx + kW - 1) / kW, ring_cols = (C->nx + 255) / 256 * 256;
  const int nrows = C->walls ? C->ny - 2 : C->ny;
  if (nodes > 1600000 && 10LL * strips * kW > 9LL * ring_cols) return;
  const int R = nodes <= (1 << 20) ? 4 : 6, bands = (nrows + R - 1) / R;
  if (bands > 65535) return;  // grid.y
  C->tile_rows = R;
  C->tile_w = kW;
  C->tile_stages = 0;
  C->tile_blocks = strips * bands;
}

cudaError_t lbm_tile_step(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches) {
  lbm_fused_args P = lbm_make_fused_args(C);
  P.fout = (float *)dst;
  P.pdl = !C->capturing;
  const dim3 grid((C->nx + kW - 1) / kW, (P.nrows + C->tile_rows - 1) / C->tile_rows);
  // One after the other on a stream, plain launches of a short kernel are 4.1 us
  // apart and programmatically dependent ones 1.5 us; captured ones 1.3 us with
  // plain graph edges, which they keep (400 x 200 step without graphs: 6.2 ->
  // 3.75 us).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((C->tile_rows + 3) * 32);
  cfg.stream = C->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = P.pdl;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel_ptr(C), (const float *)src, P);
  ++*launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}
