// lbm_internal.h -- private declarations shared by the liblbm translation units.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include "../../include/lbm.h"

// NVTX range over a scope (the library's entry points), so that a profiler
// timeline shows which call launched which kernels; free without a tool.
struct LbmRange {
  explicit LbmRange(const char *name) { nvtxRangePushA(name); }
  ~LbmRange() { nvtxRangePop(); }
  LbmRange(const LbmRange &) = delete;
  LbmRange &operator=(const LbmRange &) = delete;
};

// Device-side model constants, passed by value to every kernel.
// The EOS and model parameters are kept in double; kernels of the float
// instantiation convert them once per thread.
struct lbm_dev_params {
  int nx, ny;
  int walls;      // 1: rows 0 and ny-1 solid; 0: periodic in y as well
  int eos_kind;
  double a, b, R, T;
  double thv, thm, thl, r1, r2;
  double A, kappa, Gw;
  double s[9];    // rates in moment order (rho, e, eps, jx, qx, jy, qy, pxx, pxy)
  int n_iter, wetting;
  double rho_max;     // instability bound; psi = U = 0 at and above it
  double ghost_max;   // upper clamp of the ghost densities (<= rho_max)
};

// Per-wall-node coefficients of Eqs. 19-21, computed on the host:
// c = sin(pi/2 - theta), cot = tan(pi/2 - theta); [0..nx) bottom, [nx..2nx) top.
struct lbm_wall_coeffs {
  const double *c;
  const double *cot;
};

struct lbm_ctx {
  int nx, ny, walls, precision;
  int kernel_req, kernel_in_use;
  lbm_eos eos;
  double T, tau;
  lbm_params params;
  lbm_dev_params dp;
  double rho_v, rho_l, rho_max, rho_mid, ghost_max;
  cudaStream_t stream;
  int owns_state;
  void *state;           // two [9][ny][nx] arrays, contiguous
  void *f[2];
  int cur;               // index of the array holding the current state
  long long steps;
  unsigned long long launches;
  int status;            // sticky failure
  // device scratch
  double *d_coef;        // 4*nx: c_bot, c_top, cot_bot, cot_top
  double *d_dcoef;       // 4*nx: their derivatives in theta (adjoint)
  struct lbm_tape *tape; // adjoint record (lbm_adjoint.cu); NULL when none
  int *d_flag;           // [0]: instability, [1]: timeout, [2]: lbm_set_rho input check, [3]: arrivals of a reduction
  double *d_rho64;       // nx*ny, measurement density
  cudaStream_t xfer;     // lbm_get_rho: copy stream and its chunk events (lazy; NULL until first needed)
  cudaEvent_t xfer_ev[8];
  void *d_fields;        // 3*nx*ny reals: rho, psi, U (FP64 adjoint; lazy)
  double *d_aux;         // 8*nx*ny doubles for lbm_get_u / lbm_get_fields (lazy)
  double *d_red;         // reduction partials (red_len)
  double *d_res;         // small results
  int red_len;
  // fused kernel plan
  int fused_ok, fused_unit;  // fused kernel usable; unit-rate specialisation
  int fused_cols;            // columns per thread of the fused kernel
  int tile_rows;             // rows per tile of the small-domain kernel, 0: the ring kernel runs
  int tile_pairs;            // it also has a form that makes two steps per launch
  int tile_w, tile_blocks, tile_stages, fused_smem;
  unsigned char tmaps[4][128];   // CUtensorMap for f[0], f[1]: main box, halo box
  // lbm_step graphs, captured at the first lbm_step for both starting arrays:
  // graph_len[0] = graph_steps (even), then every power of two 2 <= 2^k below
  // it, largest first, so that any step count replays as whole graphs plus at
  // most one direct launch
  static constexpr int kMaxGraphs = 17;
  int ngraph, graphs_ready;
  int capturing;             // the library is recording launches of this context into a graph
  int graph_len[kMaxGraphs];
  cudaGraphExec_t step_graph[2][kMaxGraphs];
};

// ---- lbm_ref.cu: fields and initial states in the canonical order -----------
// All launchers return the cudaError_t of the launch and add the number of
// kernels launched to *launches.
// rho, psi, U of an FP64 state, ghost values included (the adjoint's reverse step)
cudaError_t lbm_ref_fields(const lbm_ctx *C, const double *f, double *fields, unsigned long long *launches);
// f := f_eq(rho, 0) from device or mapped host densities; with bad != NULL,
// *bad |= 1 if a fluid-node density is not finite or not > 0 (bad zeroed by
// the caller; f is written all the same)
cudaError_t lbm_ref_set_rho(const lbm_ctx *C, const double *rho, void *f, int *bad, unsigned long long *launches);
cudaError_t lbm_ref_droplets(const lbm_ctx *C, int n, const double *drop, double width, double *rho,
                             unsigned long long *launches);

// ---- lbm_api.cu -------------------------------------------------------------
// `count` steps of a context from array f[start] with its own kernel
cudaError_t lbm_launch_steps(lbm_ctx *C, int start, int count, unsigned long long *launches);

// ---- lbm_canon.cu: one step in the canonical evaluation order ---------------
cudaError_t lbm_canon_step(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches);
// Fields of the state f as doubles, [ny][nx] each: rho, psi, U (ghost values on
// the solid rows), ux, uy, Fx, Fy, Qxx, Qyy, Qxy (0 there); NULL: not wanted.
cudaError_t lbm_canon_fields(const lbm_ctx *C, const void *f, double *const (&o)[10], unsigned long long *launches);
// Largest |u|^2 over the fluid nodes.
cudaError_t lbm_canon_max_speed2(const lbm_ctx *C, const void *f, double *max2, unsigned long long *launches);

// ---- lbm_fused.cu: single-pass FP32 step ------------------------------------
int lbm_fused_plan(lbm_ctx *C);  // sets fused_ok, tile_*, tensor maps
cudaError_t lbm_fused_step(lbm_ctx *C, int src, unsigned long long *launches);
// The same step between any two state arrays of the context's shape (16-byte
// aligned): the adjoint's recorded forward and its segment replays.
cudaError_t lbm_fused_step_between(lbm_ctx *C, const void *src, void *dst, unsigned long long *launches);

// ---- lbm_tile.cu: the FP32 step of small domains ------------------------------
void lbm_tile_plan(lbm_ctx *C);  // sets tile_rows (0: not for this domain) and the tile_* shape
cudaError_t lbm_tile_step(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches);
// two steps in one launch (tile_pairs)
cudaError_t lbm_tile_pair(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches);

// ---- lbm_adjoint.cu: discrete adjoint ---------------------------------------
void lbm_adjoint_free_tape(lbm_ctx *C);

// ---- lbm_measure.cu: reductions -------------------------------------------
// n values between FP32 and double
cudaError_t lbm_widen(const lbm_ctx *C, const float *in, double *out, size_t n, unsigned long long *launches);
cudaError_t lbm_narrow(const lbm_ctx *C, const double *in, float *out, size_t n, unsigned long long *launches);
cudaError_t lbm_rho64(const lbm_ctx *C, const void *f, double *rho, unsigned long long *launches);
// the same for rows [row0, row1) only (rho indexed like the whole field)
cudaError_t lbm_rho64_rows(const lbm_ctx *C, const void *f, double *rho, int row0, int row1,
                           unsigned long long *launches);
// sum of rows [row0, row1) of a node field, in a fixed order
cudaError_t lbm_reduce_rows(const lbm_ctx *C, const double *v, int row0, int row1, double *res,
                            unsigned long long *launches);
// sum of rho over the fluid nodes of a state
cudaError_t lbm_mass_of(const lbm_ctx *C, const void *f, double *res, unsigned long long *launches);
// Apparent contact angle of the droplet on `wall` in columns [x0, x1) of the
// state f: the kernel finds where the contour cuts the boundary row and the
// centre column, lbm_angle_of interpolates there.
struct lbm_angle_cut {
  int contact;                 // 1: cuts found, 0: no contact line, -1: columns tie, lbm_angle_ties decides
  int xl, xr, steps;           // cuts right of xl and of xr, and above row `steps` from the boundary row
  double rho[6];               // at xl, xl + 1; xr, xr + 1; the last liquid node up the centre column, the next
};
struct lbm_angle_args {
  const void *f;
  int nx, ny, wall, x0, x1;
  double rho_mid;
  double *partial;    // scratch: a row of x1 - x0 doubles per chunk of rows
  unsigned *counter;  // 0 before and after
  lbm_angle_cut *res;
};
lbm_angle_args lbm_make_angle_args(const lbm_ctx *C, int wall, int x0, int x1, void *res);
// LBM_OK with the angle, height and base width, or LBM_ENOCONTACT
int lbm_angle_of(const lbm_angle_cut &r, double rho_mid, double *theta, double *H, double *L);
int lbm_angle_blocks(const lbm_angle_args &A);
cudaError_t lbm_angle(const lbm_ctx *C, const lbm_angle_args &A, unsigned long long *launches);
// the cuts of a domain that lbm_angle or lbm_angle_many left undecided
cudaError_t lbm_angle_ties(const lbm_ctx *C, const lbm_angle_args &A, unsigned long long *launches);
// the same for entries [first, first + count) (at most 65535) of a device table
// of FP32 domains; blocks: the largest lbm_angle_blocks among them
cudaError_t lbm_angle_many(const lbm_angle_args *tab, int first, int count, int blocks, cudaStream_t stream);
