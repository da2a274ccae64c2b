// lbm_ref_node.cuh -- per-node arithmetic in the canonical order (model
// constants, EOS, ghost rule), shared by the field kernels
// (lbm_ref.cu) and the adjoint kernels (lbm_adjoint.cu), which recompute the
// forward quantities of a step.  Both translation units are compiled with
// -fmad=false.
#pragma once

#include <math.h>

#include "lbm_internal.h"

namespace lbm_ref {

// D2Q9 velocities, opposite directions, the moment basis (rho, e, eps, jx, qx,
// jy, qy, pxx, pxy) and its row norms.  Kept as local tables so that fully
// unrolled loops fold every coefficient into the instruction stream.
__device__ __forceinline__ int EX(int a) {
  const int t[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
  return t[a];
}
__device__ __forceinline__ int EY(int a) {
  const int t[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
  return t[a];
}
__device__ __forceinline__ int OPP(int a) {
  const int t[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
  return t[a];
}
__device__ __forceinline__ double MC(int k, int a) {
  const double t[9][9] = {
      {1, 1, 1, 1, 1, 1, 1, 1, 1},     {-4, -1, -1, -1, -1, 2, 2, 2, 2}, {4, -2, -2, -2, -2, 1, 1, 1, 1},
      {0, 1, 0, -1, 0, 1, -1, -1, 1},  {0, -2, 0, 2, 0, 1, -1, -1, 1},   {0, 0, 1, 0, -1, 1, 1, -1, -1},
      {0, 0, -2, 0, 2, 1, 1, -1, -1},  {0, 1, -1, 1, -1, 0, 0, 0, 0},    {0, 0, 0, 0, 0, 1, -1, 1, -1}};
  return t[k][a];
}
__device__ __forceinline__ double NRM(int k) {
  const double t[9] = {9, 36, 36, 6, 12, 6, 12, 4, 4};
  return t[k];
}

// The model constants in the kernels' precision, rounded once on the host and
// passed by value: converted in the kernel, the two dozen double constants
// cost every thread of a float kernel as many instructions of the FP64 pipe
// (2 lanes per clock and SM), more than its arithmetic.
template <typename R>
struct Mdl {
  int nx, ny, walls, kind, n_iter, wetting;
  R a, b, Rg, T, thv, thm, thl, r1, r2, A, kappa, Gw, rho_max, ghost_max;
  R s[9];
  explicit Mdl(const lbm_dev_params &P)
      : nx(P.nx), ny(P.ny), walls(P.walls), kind(P.eos_kind), n_iter(P.n_iter), wetting(P.wetting),
        a((R)P.a), b((R)P.b), Rg((R)P.R), T((R)P.T), thv((R)P.thv), thm((R)P.thm), thl((R)P.thl),
        r1((R)P.r1), r2((R)P.r2), A((R)P.A), kappa((R)P.kappa), Gw((R)P.Gw), rho_max((R)P.rho_max),
        ghost_max((R)P.ghost_max) {
    for (int k = 0; k < 9; ++k) s[k] = (R)P.s[k];
  }
  __device__ bool solid_row(int y) const { return walls && (y == 0 || y == ny - 1); }
  __device__ int wx(int x) const { return x < 0 ? x + nx : (x >= nx ? x - nx : x); }
  __device__ int wy(int y) const { return y < 0 ? y + ny : (y >= ny ? y - ny : y); }
};

// Carnahan-Starling or Eq. 11 pressure.
template <typename R>
__device__ R pressure(const Mdl<R> &m, R rho) {
  if (m.kind == LBM_EOS_CARNAHAN_STARLING) {
    R eta = (m.b * rho) * (R)0.25;
    R num = (((R)1 + eta) + eta * eta) - (eta * eta) * eta;
    R den = (((R)1 - eta) * ((R)1 - eta)) * ((R)1 - eta);
    return (((rho * m.Rg) * m.T) * num) / den - (m.a * rho) * rho;
  }
  if (rho <= m.r1) return rho * m.thv;
  if (rho <= m.r2) return m.r1 * m.thv + (rho - m.r1) * m.thm;
  return (m.r1 * m.thv + (m.r2 - m.r1) * m.thm) + (rho - m.r2) * m.thl;
}

// Eq. 10 with c = 1, G = -1: U = p - rho/3, psi = sqrt(max(0, -2U)).
template <typename R>
__device__ void psi_U(const Mdl<R> &m, R rho, R &psi, R &U) {
  R u = pressure(m, rho) - rho / (R)3;
  U = u;
  psi = sqrt(fmax((R)0, (R)-2 * u));
}

// rho at node i: f_0 + f_1 + ... + f_8, left to right.
template <typename R>
__device__ __forceinline__ R node_rho(const R *__restrict__ f, size_t n, size_t i) {
  R r = (R)0;
#pragma unroll
  for (int a = 0; a < 9; ++a) r = r + f[a * n + i];
  return r;
}

// Ghost density of Eqs. 19-21 at column x of a wall, clamped: from the boundary
// row at x - 1, x, x + 1, the second row at x, c = sin(pi/2 - theta) and
// cot = tan(pi/2 - theta).
template <typename R>
__device__ __forceinline__ R ghost_rho(const Mdl<R> &m, R rim1, R ri1, R rip1, R ri2, R c, R cot) {
  const R a = rip1 - rim1;
  R g = ri2;
  if (m.n_iter <= 0) {
    g = ri2 + cot * fabs(a);
  } else {
    R d = (R)2 * (ri2 - ri1);
    for (int k = 0; k < m.n_iter; ++k) {
      R s = a * a + d * d;
      g = ri2 + c * sqrt(s);
      d = ri2 - g;
    }
  }
  return fmin(fmax(g, (R)0), m.ghost_max);
}

template <typename R>
__device__ __forceinline__ R wgt(int a) { return a <= 4 ? (R)1 / (R)3 : (R)1 / (R)12; }

// Neighbour indices of node (x, y) of a whole field [ny][nx].
template <typename R>
struct FieldNb {
  const Mdl<R> &m;
  int y, x;
  __device__ __forceinline__ size_t operator()(int ex, int ey) const {
    return (size_t)m.wy(y + ey) * m.nx + m.wx(x + ex);
  }
};

}  // namespace lbm_ref
