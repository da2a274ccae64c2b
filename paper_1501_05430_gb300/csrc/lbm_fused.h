// lbm_fused.h -- what the two kernels of the FP32 step (lbm_fused.cu: ring of
// TMA stages, for large domains; lbm_tile.cu: one tile per CTA, for small ones)
// share: their launch arguments.
#pragma once

#include <math.h>

#include "lbm_internal.h"
#include "lbm_node.cuh"

struct lbm_fused_args {
  int nx, ny, walls, wetting, n_iter, kind;
  int nstrips, nrows, y0;
  long long total;
  int stages;
  float b4, RT2, a2, r1, r2, pc0, pc1, pc2;    // EOS constants (b/4, -2RT, 2a; Eq. 11 break-
                                                // points and slopes folded into -2U)
  float A, omA, pre, halfA, rho_max, ghost_max; // force / Q constants, bounds
  lbm_node::RateK k;                            // relaxation constants
  float Gw;
  long long eoff[9];  // byte offset of plane a's destination from (row y, column x) of plane 0 for an
                      // interior node: 4 (a n + e_ay nx + e_ax) (streaming without wrap or bounce-back)
  const double *coef;
  float *fout;
  int *flag;
  int pdl;  // tile kernels: launched as a programmatic dependent
};

// Launch arguments of a context's step (all but the destination array).
inline lbm_fused_args lbm_make_fused_args(const lbm_ctx *C) {
  lbm_fused_args P;
  const lbm_dev_params &D = C->dp;
  const int W = C->tile_w;
  P.nx = C->nx;
  P.ny = C->ny;
  P.walls = C->walls;
  P.wetting = D.wetting;
  P.n_iter = D.n_iter;
  P.kind = D.eos_kind;
  P.nstrips = (C->nx + W - 1) / W;
  P.nrows = C->walls ? C->ny - 2 : C->ny;
  P.y0 = C->walls ? 1 : 0;
  P.total = (long long)P.nstrips * P.nrows;
  P.stages = C->tile_stages;
  P.pdl = 0;
  P.b4 = (float)(0.25 * D.b);
  P.RT2 = (float)(-2.0 * D.R * D.T);
  P.a2 = (float)(2.0 * D.a);
  P.r1 = (float)D.r1;
  P.r2 = (float)D.r2;
  P.pc0 = (float)(-2.0 * (D.thv - 1.0 / 3.0));
  P.pc1 = (float)(-2.0 * (D.thm - D.thv));
  P.pc2 = (float)(-2.0 * (D.thl - D.thm));
  P.A = (float)D.A;
  P.omA = (float)(1.0 - D.A);
  P.pre = (float)(-0.5 * D.kappa);
  P.halfA = (float)(0.5 * D.A);
  P.rho_max = (float)fmin(D.rho_max, 3.0e38);
  P.ghost_max = (float)fmin(D.ghost_max, 3.0e38);
  P.k = lbm_node::rate_consts(D.s);
  P.Gw = (float)D.Gw;
  {
    const long long n = (long long)C->nx * C->ny, nx = C->nx;
    const int ex[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, ey[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    for (int k = 0; k < 9; ++k) P.eoff[k] = 4 * (k * n + ey[k] * nx + ex[k]);
  }
  P.coef = C->d_coef;
  P.fout = nullptr;
  P.flag = C->d_flag;
  return P;
}

