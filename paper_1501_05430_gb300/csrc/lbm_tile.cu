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

namespace {

using lbm_node::add2;
using lbm_node::collide_node2;
using lbm_node::eos_node;
using lbm_node::eos_node2;
using lbm_node::ghost_rule;

constexpr int kW = 64;        // columns per tile: one warp per row, a lane owns columns t and t + 32
constexpr int kH = kW / 2;
constexpr int kWP = kH + 4;   // paired window entries i = -2 .. kH + 1 at index i + 2
constexpr int kWR = kW + 4;   // density window columns c = -2 .. kW + 1 at index c + 2

__device__ __forceinline__ float sum9(const float (&v)[9]) {
  return (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + v[8];
}

// (psi, psi^2) of column c into a window row: lane 0 of entry c and/or lane 1
// of entry c - kH
__device__ __forceinline__ void put(float2 *ps, float2 *sq, int c, float p, float q) {
  if (c <= kH + 1) {
    ps[c + 2].x = p;
    sq[c + 2].x = q;
  }
  if (c >= kH - 2) {
    ps[c - kH + 2].y = p;
    sq[c - kH + 2].y = q;
  }
}

// Tile of kW columns x R rows per CTA of R + 3 warps.  Warps 0 .. R + 1 each
// load one row (the tile's and the one above and below), lane t columns t and
// t + kH; the last warp loads the columns beside the tile.  Window row w holds
// row y0 - 1 + w.
template <bool UNIT, int MCW, int KIND, int R>
__global__ void __launch_bounds__((R + 3) * 32) k_tile(const float *__restrict__ fin, lbm_fused_args P) {
  static_assert(2 * (R + 2) + 4 <= 32, "one warp loads the columns beside the tile");
  __shared__ float2 wpsi[R + 2][kWP], wsq[R + 2][kWP];
  __shared__ float wrho[R + 2][kWR];
  if (P.pdl) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = blockIdx.x * kW, wr = min(kW, P.nx - x0);
  const int y0 = P.y0 + (int)blockIdx.y * R;
  const int nr = min(R, P.y0 + P.nrows - y0);  // rows of this tile
  const size_t n = (size_t)P.nx * P.ny;
  const bool geo = MCW == 0 && P.walls;
  const bool low = geo && y0 == 1, high = geo && y0 + nr == P.ny - 1;  // the tile touches a wall with a ghost row
  bool bad = false;

  // the window row and columns of this thread
  int w = warp, hc = 0;
  bool on = true;
  if (warp == R + 2) {
    const int k = lane - 2 * (R + 2);
    w = lane >> 1;
    hc = lane & 1 ? wr : -1;
    if (k >= 0) {  // densities two columns out, which the ghost values one column out read
      w = k >> 1 ? nr : 1;
      hc = k & 1 ? wr + 1 : -2;
      on = k < 4 && (k >> 1 ? high : low);
    }
  }
  on = on && w <= nr + 1;
  const int v = y0 - 1 + w;                                       // may be -1 or ny in a periodic box
  const bool solid = P.walls && (v == 0 || v == P.ny - 1);
  const int y = v < 0 ? v + P.ny : (v >= P.ny ? v - P.ny : v);
  const int c0 = lane, c1 = lane + kH;
  const bool act0 = c0 < wr, act1 = c1 < wr;  // act1 implies act0
  int gx = x0 + hc;
  gx = gx < 0 ? gx + P.nx : (gx >= P.nx ? gx - P.nx : gx);

  // the wall coefficients of a ghost row, loaded before the densities it waits for
  double k0 = 0.0, k1 = 0.0;
  if (on && solid && geo) {
    const double *coef = P.coef + (P.n_iter > 0 ? 0 : 2 * P.nx) + (v != 0 ? P.nx : 0);
    if (warp < R + 2) {
      if (act0) k0 = coef[x0 + c0];
      if (act1) k1 = coef[x0 + c1];
    } else {
      k0 = coef[gx];
    }
  }
  // a direct launch is a programmatic dependent of the step before it: from
  // here on its stores are visible
  if (P.pdl) asm volatile("griddepcontrol.wait;" ::: "memory");
  float2 f[9], r = make_float2(0.0f, 0.0f);
  if (on && warp < R + 2) {
    if (!solid) {
      if (act0) {
        const float *q0 = fin + (size_t)y * P.nx + x0 + c0, *q1 = act1 ? q0 + kH : q0;
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = make_float2(q0[a * n], q1[a * n]);
        r = add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])), add2(add2(f[4], f[5]), add2(f[6], f[7]))), f[8]);
        float2 ps, ps2;
        eos_node2<KIND>(P, r, ps, ps2);
        // unstable unless 0 < rho <= rho_max, tested on the bits
        const unsigned mx = __float_as_uint(P.rho_max);
        bad = (__float_as_uint(r.x) - 1u >= mx) | (__float_as_uint(r.y) - 1u >= mx);
        put(wpsi[w], wsq[w], c0, ps.x, ps2.x);
        wrho[w][c0 + 2] = r.x;
        if (act1) {
          put(wpsi[w], wsq[w], c1, ps.y, ps2.y);
          wrho[w][c1 + 2] = r.y;
        }
      }
    } else if (!geo) {  // Martys-Chen: psi = U = 0 on the solid rows
      put(wpsi[w], wsq[w], c0, 0.0f, 0.0f);
      put(wpsi[w], wsq[w], c1, 0.0f, 0.0f);
    }
  } else if (on) {
    if (!solid) {
      const float *q = fin + (size_t)y * P.nx + gx;
      float g[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) g[a] = q[a * n];
      const float4 e = eos_node<KIND>(P, sum9(g));
      wrho[w][hc + 2] = e.x;
      put(wpsi[w], wsq[w], hc, e.y, e.z);
    } else if (!geo) {
      put(wpsi[w], wsq[w], hc, 0.0f, 0.0f);
    }
  }
  __syncthreads();
  if (low || high) {  // uniform in the CTA
    if (on && solid) {
      // Eqs. 19-21 ghost row: v == 0 from window rows 1, 2; v == ny - 1 from the two rows below it
      const float *r1 = wrho[v != 0 ? w - 1 : 1], *r2 = wrho[v != 0 ? w - 2 : 2];
      auto ghost = [&](int c, double k) {
        const float4 e = ghost_rule<KIND>(P, r1[c + 1], r1[c + 2], r1[c + 3], r2[c + 2], (float)k, (float)k);
        put(wpsi[w], wsq[w], c, e.y, e.z);
      };
      if (warp < R + 2) {
        if (act0) ghost(c0, k0);
        if (act1) ghost(c1, k1);
      } else {
        ghost(hc, k0);
      }
    }
    __syncthreads();
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0 && *(volatile int *)P.flag == 0) atomicOr(P.flag, 1);
  if (warp < 1 || warp > nr || !act0) return;

  // collide row y (its populations are in this warp's registers)
  const float2 *pm = wpsi[w - 1], *p0 = wpsi[w], *pp = wpsi[w + 1];
  const float2 *qm = wsq[w - 1], *q0 = wsq[w], *qp = wsq[w + 1];
  const int i = lane + 2;
  const float2 pn[9] = {p0[i], p0[i + 1], pp[i], p0[i - 1], pm[i], pp[i + 1], pp[i - 1], pm[i - 1], pm[i + 1]};
  const float2 qn[9] = {q0[i], q0[i + 1], qp[i], q0[i - 1], qm[i], qp[i + 1], qp[i - 1], qm[i - 1], qm[i + 1]};
  float2 fs[9];
  collide_node2<UNIT, MCW>(P, f, pn, qn, r, y, fs);
  const bool wall_dn = P.walls && y == 1, wall_up = P.walls && y == P.ny - 2;
  const unsigned nx = P.nx, un = (unsigned)n;
  const unsigned ry = (unsigned)y * nx, rym = (unsigned)(y == 0 ? P.ny - 1 : y - 1) * nx,
                 ryp = (unsigned)(y == P.ny - 1 ? 0 : y + 1) * nx;
  float *const o0 = P.fout, *const o1 = o0 + un, *const o2 = o1 + un, *const o3 = o2 + un, *const o4 = o3 + un;
  float *const o5 = o4 + un, *const o6 = o5 + un, *const o7 = o6 + un, *const o8 = o7 + un;
  // streaming with half-way bounce-back of node x's post-collision populations
  auto push = [&](unsigned x, float f0, float f1, float f2, float f3, float f4, float f5, float f6, float f7,
                  float f8) {
    const unsigned xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    o0[ry + x] = f0;
    o1[ry + xp] = f1;
    o3[ry + xm] = f3;
    if (wall_up) {
      o4[ry + x] = f2;
      o7[ry + x] = f5;
      o8[ry + x] = f6;
    } else {
      o2[ryp + x] = f2;
      o5[ryp + xp] = f5;
      o6[ryp + xm] = f6;
    }
    if (wall_dn) {
      o2[ry + x] = f4;
      o5[ry + x] = f7;
      o6[ry + x] = f8;
    } else {
      o4[rym + x] = f4;
      o7[rym + xm] = f7;
      o8[rym + xp] = f8;
    }
  };
  push(x0 + c0, fs[0].x, fs[1].x, fs[2].x, fs[3].x, fs[4].x, fs[5].x, fs[6].x, fs[7].x, fs[8].x);
  if (act1) push(x0 + c1, fs[0].y, fs[1].y, fs[2].y, fs[3].y, fs[4].y, fs[5].y, fs[6].y, fs[7].y, fs[8].y);
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
