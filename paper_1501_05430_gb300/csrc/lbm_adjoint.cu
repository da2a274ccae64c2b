// lbm_adjoint.cu -- discrete adjoint (reverse-time) of the reference step.
//
// Forward step n -> n+1 (lbm_ref.cu): rho, psi, U (Eqs. 1, 10-11); ghost rows
// (Eqs. 19-21); per fluid node the force F (Eq. 9 [+ Eq. 14]) and tensor Q
// (Eq. 17) from the 3x3 stencil of (psi, U); the MRT collision with Guo
// forcing and the Eq. 16 source (Eqs. 4-6, 15); push streaming with half-way
// bounce-back.  Given lam = dL/df^{n+1}, one reverse step computes
// dL/df^n and adds this step's part of dL/dtheta (per wall node, through
// c = sin(pi/2 - theta) of Eq. 21 or cot of Eq. 19) and dL/dT (through the
// EOS), in FP32 in one kernel (k_adj_step), in FP64 in four (after the fields):
//
//   k_adj_collide  per fluid node: pull lam back through the streaming
//                  (bounce-back included), recompute F, Q and the collision,
//                  and transpose it: dL/df through the moments, velocity,
//                  equilibrium and forcing, plus dL/dF and dL/dQ (5 values).
//   k_adj_psi      per node (ghost rows too): gather dL/dpsi and dL/dU from
//                  the dL/dF, dL/dQ of the fluid nodes whose stencil holds it
//                  (its own included), map them to dL/drho through the EOS
//                  (psi = sqrt(-2U): dpsi/dU = -1/psi, 0 where psi = 0) and
//                  add the node's dL/dT.
//   k_adj_ghost    per wall node: back through the clamp and the n_iter
//                  iterations of Eq. 20 (or Eq. 19) to the densities of the
//                  boundary row (x-1, x, x+1) and the second row, and to theta.
//   k_adj_finish   per fluid node: dL/df^n_a = collision part + dL/drho for
//                  every a (rho = sum_a f_a), the ghost-rule parts gathered
//                  from the neighbouring wall nodes.
//
// Kinks follow the oracle's convention: d sqrt(s)/ds = 0 at s = 0, d|a|/da = 0
// at a = 0, clamped ghost densities pass nothing.  Gathers instead of atomics
// keep every sum in a fixed order (the result is reproducible bit for bit).
//
// Recording: lbm_adjoint_record runs the steps with the context's own step
// kernel and keeps the state every `checkpoint_every` steps;
// lbm_adjoint_backward replays each segment forward with the same kernel into
// a segment buffer and then walks it back (the canonical fields of each
// state, ghost rows included, are recomputed first).
#include <math.h>
#include <string.h>

#include <new>
#include <vector>

#include "lbm_internal.h"
#include "lbm_ref_node.cuh"

using namespace lbm_ref;

struct lbm_tape {
  int nsteps, every, nseg;
  size_t state_bytes;            // one [9][ny][nx] array
  std::vector<void *> ckpt;      // state at the start of each segment
  void *seg;                     // (every + 1) states of the segment being reversed
  void *lam[2];                  // adjoint fields
  void *aux;                     // FP64: 5 planes: dL/dFx, dL/dFy, dL/dQxx, dL/dQyy, dL/dQxy
  void *rhob;                    // FP64: dL/drho per node (ghost rows: of the ghost density)
  double *tacc;                  // per-node dL/dT, accumulated over the steps
  double *gpart;                 // FP64: [2 walls][4][nx]: ghost-rule partials
  double *dtheta;                // [2][nx]
  double *red;                   // reduction output
  // captured graphs (contexts with a non-NULL stream): the recorded forward of
  // one full segment per starting array, and the replay + reverse sweep of one
  // full segment per starting adjoint buffer
  cudaGraphExec_t fwd_graph[2], bwd_graph[2];
  unsigned long long fwd_launches, bwd_launches;  // kernels per replay
};

namespace {

constexpr int kMaxIter = 64;

template <typename R>
__device__ void eos_derivs(const Mdl<R> &m, R rho, R &dp_drho, R &dp_dT) {
  if (m.kind == LBM_EOS_CARNAHAN_STARLING) {
    // p = rho R T Z(eta) - a rho^2, Z = N/D, N = 1 + eta + eta^2 - eta^3, D = (1 - eta)^3, eta = b rho/4:
    // dp/drho = R T (Z + eta dZ/deta) - 2 a rho,  dZ/deta = N'/D + 3 N/(1 - eta)^4
    R eta = (m.b * rho) * (R)0.25;
    R om = (R)1 - eta;
    R num = (((R)1 + eta) + eta * eta) - (eta * eta) * eta;
    R dnum = ((R)1 + (R)2 * eta) - (R)3 * (eta * eta);
    R den = (om * om) * om;
    R Z = num / den;
    R dZ = dnum / den + ((R)3 * num) / (den * om);
    dp_drho = (m.Rg * m.T) * (Z + eta * dZ) - (R)2 * (m.a * rho);
    dp_dT = (rho * m.Rg) * Z;
  } else {
    dp_dT = (R)0;
    dp_drho = rho <= m.r1 ? m.thv : (rho <= m.r2 ? m.thm : m.thl);
  }
}

// Transpose of the collision at one fluid node: from ls = dL/df* (pulled back
// through the streaming), the populations f, rho and F to the part of dL/df that
// passes through the moments (cl), and aux = dL/d(Fx, Fy, Qxx, Qyy, Qxy).
template <typename R>
__device__ __forceinline__ void adj_collide(const Mdl<R> &m, const R (&f)[9], const R (&ls)[9], R rho, R Fx, R Fy,
                                            R (&cl)[9], R (&aux)[5]) {
  R mm[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    R acc = (R)0;
#pragma unroll
    for (int a = 0; a < 9; ++a)
      if (MC(k, a) != 0.0) acc = acc + (R)MC(k, a) * f[a];
    mm[k] = acc;
  }
  const R vx = (mm[3] + (R)0.5 * Fx) / rho, vy = (mm[5] + (R)0.5 * Fy) / rho;
  const R v2 = vx * vx + vy * vy;
  // f* = M^T diag(1/N) m*  ->  dL/dm*_k = sum_a M_ka ls_a / N_k
  R msb[9], mb[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    R acc = (R)0;
#pragma unroll
    for (int a = 0; a < 9; ++a)
      if (MC(k, a) != 0.0) acc = acc + (R)MC(k, a) * ls[a];
    msb[k] = acc / (R)NRM(k);
  }
  // m*_k = m_k - s_k (m_k - meq_k) + (1 - s_k/2) S_k + C_k
  R meqb[9], Sb[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    mb[k] = ((R)1 - m.s[k]) * msb[k];
    meqb[k] = m.s[k] * msb[k];
    Sb[k] = ((R)1 - (R)0.5 * m.s[k]) * msb[k];
  }
  // C_1 = 1.5 s_1 (Qxx + Qyy), C_7 = -s_7 (Qxx - Qyy), C_8 = -s_8 Qxy
  const R Qxxb = ((R)1.5 * m.s[1]) * msb[1] - m.s[7] * msb[7];
  const R Qyyb = ((R)1.5 * m.s[1]) * msb[1] + m.s[7] * msb[7];
  const R Qxyb = -(m.s[8] * msb[8]);
  // S = (0, 6 vF, -6 vF, Fx, -Fx, Fy, -Fy, 2 (vx Fx - vy Fy), vx Fy + vy Fx), vF = v.F
  const R vFb = (R)6 * (Sb[1] - Sb[2]);
  R Fxb = (Sb[3] - Sb[4]) + (R)2 * vx * Sb[7] + vy * Sb[8] + vx * vFb;
  R Fyb = (Sb[5] - Sb[6]) - (R)2 * vy * Sb[7] + vx * Sb[8] + vy * vFb;
  R vxb = (R)2 * Fx * Sb[7] + Fy * Sb[8] + Fx * vFb;
  R vyb = -((R)2 * Fy * Sb[7]) + Fx * Sb[8] + Fy * vFb;
  // meq = rho (1, -2 + 3 v2, 1 - 3 v2, vx, -vx, vy, -vy, vx^2 - vy^2, vx vy)
  R rhob = meqb[0] + meqb[1] * ((R)-2 + (R)3 * v2) + meqb[2] * ((R)1 - (R)3 * v2) + (meqb[3] - meqb[4]) * vx +
           (meqb[5] - meqb[6]) * vy + meqb[7] * (vx * vx - vy * vy) + meqb[8] * (vx * vy);
  const R v2b = (R)3 * rho * (meqb[1] - meqb[2]);
  vxb = vxb + (R)2 * vx * v2b + rho * (meqb[3] - meqb[4]) + (R)2 * rho * vx * meqb[7] + rho * vy * meqb[8];
  vyb = vyb + (R)2 * vy * v2b + rho * (meqb[5] - meqb[6]) - (R)2 * rho * vy * meqb[7] + rho * vx * meqb[8];
  // v = (j + F/2) / rho
  mb[3] = mb[3] + vxb / rho;
  mb[5] = mb[5] + vyb / rho;
  Fxb = Fxb + (R)0.5 * vxb / rho;
  Fyb = Fyb + (R)0.5 * vyb / rho;
  rhob = rhob - (vxb * vx + vyb * vy) / rho;
  // m = M f and rho = sum_a f_a
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    R acc = rhob;
#pragma unroll
    for (int k = 0; k < 9; ++k)
      if (MC(k, a) != 0.0) acc = acc + (R)MC(k, a) * mb[k];
    cl[a] = acc;
  }
  aux[0] = Fxb;
  aux[1] = Fyb;
  aux[2] = Qxxb;
  aux[3] = Qyyb;
  aux[4] = Qxyb;
}

// dL/drho and dL/dT of node (row y) through psi and U, gathered from the aux of
// the fluid nodes whose stencils hold it; ax(ex, ey) is the index of a neighbour
// in the planes aux + k * an, nb(ex, ey) its index in psi.  rho: its density.
template <typename R, typename Nb, typename Ax>
__device__ __forceinline__ void adj_psi(const Mdl<R> &m, const R *__restrict__ psi, const R *__restrict__ aux,
                                        size_t an, int y, R rho, Nb nb, Ax ax, R &rb, double &tb) {
  const R G = (R)-1;
  const R pre = m.kappa * (G * (R)0.5);
  const R omA = (R)1 - m.A;
  const R psi_p = psi[nb(0, 0)];
  R pb = (R)0, ub = (R)0;
  // fluid nodes q = p - e_a hold p in their stencil in direction a:
  //   dF(q)/dpsi_p = (1-A) psi_q w_a e_a,  dF(q)/dU_p = -A w_a e_a,
  //   dQ_ij(q)/dpsi_p = pre w_a e_ai e_aj ((1-A) psi_q + A psi_p)
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    int yq = y - EY(a);
    if (m.walls && (yq < 0 || yq >= m.ny)) continue;
    if (m.solid_row(m.wy(yq))) continue;
    const R *q = aux + ax(-EX(a), -EY(a));
    const R w = wgt<R>(a);
    const R eF = q[0] * (R)EX(a) + q[an] * (R)EY(a);
    const R eQ = q[2 * an] * (R)(EX(a) * EX(a)) + q[3 * an] * (R)(EY(a) * EY(a)) + q[4 * an] * (R)(EX(a) * EY(a));
    const R psi_q = psi[nb(-EX(a), -EY(a))];
    pb = pb + (omA * psi_q) * w * eF + pre * w * eQ * (omA * psi_q + m.A * psi_p);
    ub = ub - m.A * w * eF;
  }
  const bool fluid = !m.solid_row(y);
  if (fluid) {
    // own terms: dF/dpsi_0 = (1-A) s_psi (+ Eq. 14), dQ_ii/dpsi_0 = pre ((1-A) q1_ii - psi_0),
    // dQ_xy/dpsi_0 = pre (1-A) q1_xy
    R spx = 0, spy = 0, ssx = 0, ssy = 0, qxx1 = 0, qyy1 = 0, qxy1 = 0;
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      const R w = wgt<R>(a);
      const R pn = psi[nb(EX(a), EY(a))];
      const R sol = m.solid_row(m.wy(y + EY(a))) ? (R)1 : (R)0;
      spx = spx + w * pn * (R)EX(a);
      spy = spy + w * pn * (R)EY(a);
      ssx = ssx + w * sol * (R)EX(a);
      ssy = ssy + w * sol * (R)EY(a);
      const R t1 = w * (pn - psi_p);
      qxx1 = qxx1 + t1 * (R)(EX(a) * EX(a));
      qyy1 = qyy1 + t1 * (R)(EY(a) * EY(a));
      qxy1 = qxy1 + t1 * (R)(EX(a) * EY(a));
    }
    const R *o = aux + ax(0, 0);
    const R Fxb = o[0], Fyb = o[an];
    pb = pb + omA * (Fxb * spx + Fyb * spy);
    if (m.wetting == LBM_WET_MARTYS_CHEN) pb = pb - m.Gw * (Fxb * ssx + Fyb * ssy);
    pb = pb + pre * (omA * (o[2 * an] * qxx1 + o[3 * an] * qyy1 + o[4 * an] * qxy1) - psi_p * (o[2 * an] + o[3 * an]));
  }
  // to dL/drho (and dL/dT) through U = p(rho) - rho/3 and psi = sqrt(-2U)
  rb = (R)0;
  tb = 0.0;
  const bool ghost = !fluid && m.wetting == LBM_WET_GEOMETRIC;
  if (fluid || (ghost && rho < m.rho_max)) {
    R dp, dpT;
    eos_derivs(m, rho, dp, dpT);
    const R ut = ub - (psi_p > (R)0 ? pb / psi_p : (R)0);
    rb = ut * (dp - (R)1 / (R)3);
    tb = (double)(ut * dpT);
  }
}

// Transpose of the ghost rule at one wall node, from gb = dL/d(its density):
// part = dL/d(rho(x-1), rho(x+1), rho(x) of the boundary row, rho(x) of the
// second row); returns dL/dtheta.  dc, dcot: derivatives of c and cot in theta.
template <typename R>
__device__ __forceinline__ double adj_ghost(const Mdl<R> &m, R rim1, R ri1, R rip1, R ri2, R c, R cot, double dc,
                                            double dcot, R gb, double (&part)[4]) {
  R a = rip1 - rim1;
  // forward again, keeping the iterates
  R d[kMaxIter];
  R g;
  const int nit = m.n_iter < kMaxIter ? m.n_iter : kMaxIter;
  if (nit <= 0) {
    g = ri2 + cot * fabs(a);
  } else {
    d[0] = (R)2 * (ri2 - ri1);
    g = ri2;
    for (int k = 0; k < nit; ++k) {
      R s = a * a + d[k] * d[k];
      g = ri2 + c * sqrt(s);
      if (k + 1 < nit) d[k + 1] = ri2 - g;
    }
  }
  if (!(g > (R)0 && g < m.ghost_max)) gb = (R)0;  // clamped: no gradient
  R ab = 0, ri1b = 0, ri2b = 0, cb = 0, cotb = 0;
  if (nit <= 0) {
    ri2b = gb;
    cotb = gb * fabs(a);
    ab = a > (R)0 ? gb * cot : (a < (R)0 ? -(gb * cot) : (R)0);
  } else {
    R gbar = gb;
    for (int k = nit - 1; k >= 0; --k) {
      // g_{k+1} = ri2 + c sqrt(a^2 + d_k^2)
      R s = a * a + d[k] * d[k];
      R sq = sqrt(s);
      ri2b = ri2b + gbar;
      cb = cb + gbar * sq;
      R sb = s > (R)0 ? (gbar * c) * (R)0.5 / sq : (R)0;
      ab = ab + sb * (R)2 * a;
      R db = sb * (R)2 * d[k];
      if (k >= 1) {  // d_k = ri2 - g_k
        ri2b = ri2b + db;
        gbar = -db;
      } else {  // d_0 = 2 (ri2 - ri1)
        ri2b = ri2b + (R)2 * db;
        ri1b = ri1b - (R)2 * db;
      }
    }
  }
  part[0] = -(double)ab;
  part[1] = (double)ab;
  part[2] = (double)ri1b;
  part[3] = (double)ri2b;
  return (double)cb * dc + (double)cotb * dcot;
}

// ---- one reverse step in one kernel -----------------------------------------------

constexpr int kTW = 32, kTH = 8;                 // largest tile
constexpr int kAW = kTW + 4, kAH = kTH + 2;      // nodes with aux: 2 columns and 1 row around the tile
constexpr int kFW = kTW + 6, kFH = kTH + 4;      // nodes with fields: 3 columns and 2 rows around it
constexpr int kStepThreads = 480;                // one node per thread in every phase

// lam_out = the reverse step of lam_in at the state f, for the tile of kTW
// columns x at most kTH rows of this CTA.  Phases, a barrier after each:
// fields (the values of k_fields) of every node in reach; the transposed
// collision of every node whose aux the tile reads (threads of the tile keep
// the part that passes through the moments in registers); dL/drho through psi
// and U, and at the ghost nodes the transpose of the ghost rule; the sums.
// Small domains are bound by the latency of a kernel, and five kernels with
// four global round trips of fields, aux and dL/drho took 19 us (captured; 28
// launched directly) where this one takes 9; its repeated work at the tiles'
// edges (1.8 times the fields, 1.4 times the collisions) is paid for at any size
// by the 170 bytes a node that are not moved: reverse step with its replay, us,
// five kernels -> one, 256 x 128 21.9 -> 12.0, 800 x 400 61 -> 55, 1600 x 800
// 245 -> 238.  In FP64 the repeated work costs more than it saves (800 x 400
// 816 -> 1040; the FP64 pipe is the limit), so FP64 keeps the kernels below.
template <typename R>
__global__ void __launch_bounds__(kStepThreads)
    k_adj_step(Mdl<R> m, int strips, int bands, const R *__restrict__ f, const R *__restrict__ lam_in,
               R *__restrict__ lam_out, const double *__restrict__ coef, const double *__restrict__ dcoef,
               double *__restrict__ tacc, double *__restrict__ dtheta, int *flag) {
  __shared__ R srho[kFH * kFW], spsi[kFH * kFW], sU[kFH * kFW];
  __shared__ R saux[5 * kAH * kAW];
  __shared__ double sgp[2][4][kAW];  // ghost-rule parts by wall, part, column (as in aux)
  const int band = (int)(blockIdx.x / (unsigned)strips);
  const int x0 = ((int)blockIdx.x - band * strips) * kTW, wr = min(kTW, m.nx - x0);
  const int first = m.walls ? 1 : 0, rows = m.walls ? m.ny - 2 : m.ny;
  // equal bands: with walls the outer ones hold both rows that a ghost node reads
  const int ya = first + (int)((long long)band * rows / bands), yb = first + (int)((long long)(band + 1) * rows / bands);
  const int hr = yb - ya;
  const size_t n = (size_t)m.nx * m.ny;
  const bool geo = m.walls && m.wetting == LBM_WET_GEOMETRIC;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // this thread's node: rows ya - 1 .. yb, columns x0 - 2 .. x0 + wr + 1
  const int cy = threadIdx.x / kAW, cx = threadIdx.x - cy * kAW, v = ya - 1 + cy;
  const bool on = cy < hr + 2 && cx < wr + 4;  // (in a walled domain all these rows exist)
  const int y = m.wy(v), x = m.wx(x0 - 2 + cx);
  const bool solid = m.solid_row(y), own = on && cx >= 2 && cx < wr + 2 && (solid || (cy >= 1 && cy <= hr));
  const size_t i = (size_t)y * m.nx + x;
  const int jf = (cy + 1) * kFW + cx + 1, ja = cy * kAW + cx;  // its place among the fields and aux
  auto nb = [&](int ex, int ey) { return jf + ey * kFW + ex; };
  auto ax = [&](int ex, int ey) { return ja + ey * kAW + ex; };
  R ls[9], fl[9], cl[9];
  if (on && !solid) {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int yt = m.wy(y + EY(a));
      ls[a] = m.solid_row(yt) ? lam_in[OPP(a) * n + i] : lam_in[a * n + (size_t)yt * m.nx + m.wx(x + EX(a))];
      fl[a] = f[a * n + i];
    }
  }
  // fields: rows ya - 2 .. yb + 1, columns x0 - 3 .. x0 + wr + 2
  bool bad = false;
  const int t = threadIdx.x, fy = t / kFW, fx = t - fy * kFW, fv = ya - 2 + fy;
  if (fy < hr + 4 && fx < wr + 6 && !(m.walls && (fv < 0 || fv >= m.ny))) {
    const int y = m.wy(fv), x = m.wx(x0 - 3 + fx);
    R r, psi = (R)0, U = (R)0;
    if (!m.solid_row(y)) {
      r = node_rho(f, n, (size_t)y * m.nx + x);
      psi_U(m, r, psi, U);
      bad |= !(r > (R)0) || r > m.rho_max;
    } else if (geo) {
      const int w = y == 0 ? 0 : 1;
      const size_t b1 = (size_t)(w == 0 ? 1 : m.ny - 2) * m.nx, b2 = (size_t)(w == 0 ? 2 : m.ny - 3) * m.nx;
      r = ghost_rho(m, node_rho(f, n, b1 + m.wx(x - 1)), node_rho(f, n, b1 + x), node_rho(f, n, b1 + m.wx(x + 1)),
                    node_rho(f, n, b2 + x), (R)coef[w * m.nx + x], (R)coef[2 * m.nx + w * m.nx + x]);
      if (r < m.rho_max) psi_U(m, r, psi, U);
    } else {
      r = (R)0;
    }
    srho[t] = r;
    spsi[t] = psi;
    sU[t] = U;
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
  if (on && !solid) {
    R Fx, Fy, Qxx, Qyy, Qxy, a5[5];
    force_Q(m, spsi, sU, y, nb, Fx, Fy, Qxx, Qyy, Qxy);
    adj_collide(m, fl, ls, srho[jf], Fx, Fy, cl, a5);
#pragma unroll
    for (int k = 0; k < 5; ++k) saux[k * kAH * kAW + ja] = a5[k];
  }
  __syncthreads();
  // dL/drho: the tile's nodes, and the ghost nodes of one more column each side
  R rb = (R)0;
  if (own || (on && solid && geo && cx >= 1 && cx < wr + 3)) {
    double tb;
    adj_psi(m, spsi, saux, kAH * kAW, y, srho[jf], nb, ax, rb, tb);
    if (own) tacc[i] += tb;
    if (solid && geo) {
      const int w = y == 0 ? 0 : 1, s = w == 0 ? kFW : -kFW;
      double part[4];
      const double dth = adj_ghost(m, srho[jf + s - 1], srho[jf + s], srho[jf + s + 1], srho[jf + 2 * s],
                                   (R)coef[w * m.nx + x], (R)coef[2 * m.nx + w * m.nx + x], dcoef[w * m.nx + x],
                                   dcoef[2 * m.nx + w * m.nx + x], rb, part);
      if (own) dtheta[w * m.nx + x] += dth;
#pragma unroll
      for (int k = 0; k < 4; ++k) sgp[w][k][cx] = part[k];
    }
  }
  if (geo && (ya == 1 || yb == m.ny - 1)) __syncthreads();
  if (!own) return;
  if (solid) {
#pragma unroll
    for (int a = 0; a < 9; ++a) lam_out[a * n + i] = (R)0;
    return;
  }
  if (geo && (y <= 2 || y >= m.ny - 3)) {
    double r = (double)rb;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int y1 = w == 0 ? 1 : m.ny - 2, y2 = w == 0 ? 2 : m.ny - 3;
      // boundary row: this node is x-1 of wall node x+1, x+1 of wall node x-1, and x of wall node x
      if (y == y1) r += sgp[w][0][cx + 1] + sgp[w][1][cx - 1] + sgp[w][2][cx];
      if (y == y2) r += sgp[w][3][cx];
    }
    rb = (R)r;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) lam_out[a * n + i] = cl[a] + rb;
}

// ---- the four kernels of a reverse step on whole fields (FP64, see reverse_step) --

template <typename R>
__global__ void k_adj_collide(Mdl<R> m, const R *__restrict__ f, const R *__restrict__ fields,
                              const R *__restrict__ lam_in, R *__restrict__ lam_out, R *__restrict__ aux) {
  size_t n = (size_t)m.nx * m.ny;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int y = (int)(i / m.nx), x = (int)(i - (size_t)y * m.nx);
  if (m.solid_row(y)) return;
  // adjoint of the post-collision populations (transpose of the push streaming)
  R ls[9], fl[9], cl[9], ax[5];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    int yt = m.wy(y + EY(a));
    ls[a] = m.solid_row(yt) ? lam_in[OPP(a) * n + i] : lam_in[a * n + (size_t)yt * m.nx + m.wx(x + EX(a))];
    fl[a] = f[a * n + i];
  }
  R Fx, Fy, Qxx, Qyy, Qxy;
  force_Q(m, fields + n, fields + 2 * n, y, FieldNb<R>{m, y, x}, Fx, Fy, Qxx, Qyy, Qxy);
  adj_collide(m, fl, ls, fields[i], Fx, Fy, cl, ax);
#pragma unroll
  for (int a = 0; a < 9; ++a) lam_out[a * n + i] = cl[a];
#pragma unroll
  for (int k = 0; k < 5; ++k) aux[k * n + i] = ax[k];
}

template <typename R>
__global__ void k_adj_psi(Mdl<R> m, const R *__restrict__ fields, const R *__restrict__ aux,
                          R *__restrict__ rhob_out, double *__restrict__ tacc) {
  size_t n = (size_t)m.nx * m.ny;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int y = (int)(i / m.nx), x = (int)(i - (size_t)y * m.nx);
  const FieldNb<R> nb{m, y, x};
  R rb;
  double tb;
  adj_psi(m, fields + n, aux, n, y, fields[i], nb, nb, rb, tb);
  rhob_out[i] = rb;
  tacc[i] += tb;
}

template <typename R>
__global__ void k_adj_ghost(Mdl<R> m, const R *__restrict__ fields, const double *__restrict__ coef,
                            const double *__restrict__ dcoef, const R *__restrict__ rhob,
                            double *__restrict__ gpart, double *__restrict__ dtheta) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2 * m.nx) return;
  int w = t / m.nx, x = t - w * m.nx;
  int yg = w == 0 ? 0 : m.ny - 1, y1 = w == 0 ? 1 : m.ny - 2, y2 = w == 0 ? 2 : m.ny - 3;
  const R *r1 = fields + (size_t)y1 * m.nx, *r2 = fields + (size_t)y2 * m.nx;
  double part[4];
  dtheta[w * m.nx + x] += adj_ghost(m, r1[m.wx(x - 1)], r1[x], r1[m.wx(x + 1)], r2[x], (R)coef[w * m.nx + x],
                                    (R)coef[2 * m.nx + w * m.nx + x], dcoef[w * m.nx + x],
                                    dcoef[2 * m.nx + w * m.nx + x], rhob[(size_t)yg * m.nx + x], part);
#pragma unroll
  for (int k = 0; k < 4; ++k) gpart[((size_t)w * 4 + k) * m.nx + x] = part[k];
}

template <typename R>
__global__ void k_adj_finish(Mdl<R> m, R *__restrict__ lam, const R *__restrict__ rhob,
                             const double *__restrict__ gpart, int geo) {
  size_t n = (size_t)m.nx * m.ny;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int y = (int)(i / m.nx), x = (int)(i - (size_t)y * m.nx);
  if (m.solid_row(y)) {
#pragma unroll
    for (int a = 0; a < 9; ++a) lam[a * n + i] = (R)0;
    return;
  }
  double r = (double)rhob[i];
  if (geo) {
    const int xm = m.wx(x - 1), xp = m.wx(x + 1);
    for (int w = 0; w < 2; ++w) {
      const double *gp = gpart + (size_t)w * 4 * m.nx;
      const int y1 = w == 0 ? 1 : m.ny - 2, y2 = w == 0 ? 2 : m.ny - 3;
      // boundary row: this node is x-1 of wall node x+1, x+1 of wall node x-1, and x of wall node x
      if (y == y1) r += gp[xp] + gp[m.nx + xm] + gp[2 * m.nx + x];
      if (y == y2) r += gp[3 * m.nx + x];
    }
  }
  const R rr = (R)r;
#pragma unroll
  for (int a = 0; a < 9; ++a) lam[a * n + i] = lam[a * n + i] + rr;
}

template <typename R>
__global__ void k_adj_init(lbm_dev_params P, const double *__restrict__ dl_drho, R *__restrict__ lam) {
  size_t n = (size_t)P.nx * P.ny;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int y = (int)(i / P.nx);
  const bool solid = P.walls && (y == 0 || y == P.ny - 1);
  const R v = solid ? (R)0 : (R)dl_drho[i];
#pragma unroll
  for (int a = 0; a < 9; ++a) lam[a * n + i] = v;
}

template <typename R>
__global__ void k_to_double(const R *__restrict__ in, double *__restrict__ out, size_t n) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (double)in[i];
}

#define ACK(x)                          \
  do {                                  \
    if ((x) != cudaSuccess) {           \
      cudaGetLastError();               \
      return LBM_ECUDA;                 \
    }                                   \
  } while (0)

size_t rsize(const lbm_ctx *C) { return C->precision == 64 ? sizeof(double) : sizeof(float); }

// One forward step src -> dst with the context's own step kernel: the fused
// FP32 kernel where the context runs it (so the recorded forward advances
// exactly like lbm_step), else the canonical kernel.  The reverse
// kernels transpose the canonical step at the states this produces.
int fwd_step(lbm_ctx *C, const void *src, void *dst) {
  if (C->kernel_in_use == LBM_KERNEL_FUSED) {
    ACK(lbm_fused_step_between(C, src, dst, &C->launches));
    return LBM_OK;
  }
  ACK(lbm_canon_step(C, src, dst, &C->launches));
  return LBM_OK;
}

template <typename R>
int reverse_step(lbm_ctx *C, lbm_tape *T, const void *f, int lin) {
  const Mdl<R> m(C->dp);
  R *lam_in = (R *)T->lam[lin], *lam_out = (R *)T->lam[lin ^ 1];
  if constexpr (sizeof(R) == sizeof(float)) {
    const int rows = C->walls ? C->ny - 2 : C->ny, strips = (C->nx + kTW - 1) / kTW, bands = (rows + kTH - 1) / kTH;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)strips * (unsigned)bands);
    cfg.blockDim = dim3(kStepThreads);
    cfg.stream = C->stream;
    // direct launches overlap their set-up with the kernel before (as k_tile's); captured ones keep plain edges
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C->capturing ? 0 : 1;
    ACK(cudaLaunchKernelEx(&cfg, k_adj_step<R>, m, strips, bands, (const R *)f, (const R *)lam_in, lam_out,
                           (const double *)C->d_coef, (const double *)C->d_dcoef, T->tacc, T->dtheta, C->d_flag));
    ++C->launches;
    return LBM_OK;
  } else {
    const int B = 256;
    const size_t n = (size_t)C->nx * C->ny;
    const unsigned g = (unsigned)((n + B - 1) / B), gw = (unsigned)((2 * C->nx + B - 1) / B);
    const R *fields = (const R *)C->d_fields;
    ACK(lbm_ref_fields(C, (const double *)f, (double *)C->d_fields, &C->launches));
    k_adj_collide<R><<<g, B, 0, C->stream>>>(m, (const R *)f, fields, lam_in, lam_out, (R *)T->aux);
    k_adj_psi<R><<<g, B, 0, C->stream>>>(m, fields, (const R *)T->aux, (R *)T->rhob, T->tacc);
    C->launches += 2;
    const int geo = C->walls && m.wetting == LBM_WET_GEOMETRIC;
    if (geo) {
      k_adj_ghost<R><<<gw, B, 0, C->stream>>>(m, fields, C->d_coef, C->d_dcoef, (const R *)T->rhob, T->gpart,
                                              T->dtheta);
      ++C->launches;
    }
    k_adj_finish<R><<<g, B, 0, C->stream>>>(m, lam_out, (const R *)T->rhob, T->gpart, geo);
    ++C->launches;
    ACK(cudaGetLastError());
    return LBM_OK;
  }
}

// Capture the work that fn() enqueues on the context stream into *out; the
// kernels it launches are counted into *launches (not into the context).
template <typename Fn>
int capture(lbm_ctx *C, cudaGraphExec_t *out, unsigned long long *launches, Fn fn) {
  cudaGraph_t graph = nullptr;
  if (cudaStreamBeginCapture(C->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
    cudaGetLastError();
    return LBM_ECUDA;
  }
  const unsigned long long l0 = C->launches;
  C->capturing = 1;
  int st = fn();
  C->capturing = 0;
  *launches = C->launches - l0;
  C->launches = l0;
  cudaError_t e = cudaStreamEndCapture(C->stream, &graph);
  if (st == LBM_OK && e == cudaSuccess) e = cudaGraphInstantiate(out, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  if (st == LBM_OK && e != cudaSuccess) st = LBM_ECUDA;
  if (st != LBM_OK) {
    cudaGetLastError();
    *out = nullptr;
  }
  return st;
}

// Replay of a segment from seg[0] (len states) and its reverse sweep, adjoint
// starting in lam[lin]; returns the status and leaves the final buffer in *lin.
template <typename R>
int segment_reverse(lbm_ctx *C, lbm_tape *T, int len, int *lin) {
  char *seg = (char *)T->seg;
  int st = LBM_OK;
  for (int k = 0; k + 1 < len && st == LBM_OK; ++k)
    st = fwd_step(C, seg + (size_t)k * T->state_bytes, seg + (size_t)(k + 1) * T->state_bytes);
  for (int k = len - 1; k >= 0 && st == LBM_OK; --k) {
    st = reverse_step<R>(C, T, seg + (size_t)k * T->state_bytes, *lin);
    *lin ^= 1;
  }
  return st;
}

template <typename R>
int backward(lbm_ctx *C, lbm_tape *T, const double *dl_drho, double *dl_dtheta, double *dl_dT, double *dl_df0) {
  const size_t n = (size_t)C->nx * C->ny;
  const int B = 256;
  double *h = nullptr;
  ACK(cudaMalloc(&h, n * sizeof(double)));
  cudaError_t e = cudaMemcpyAsync(h, dl_drho, n * sizeof(double), cudaMemcpyHostToDevice, C->stream);
  if (e == cudaSuccess) {
    k_adj_init<R><<<(unsigned)((n + B - 1) / B), B, 0, C->stream>>>(C->dp, h, (R *)T->lam[0]);
    ++C->launches;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(T->tacc, 0, n * sizeof(double), C->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(T->dtheta, 0, 2 * (size_t)C->nx * sizeof(double), C->stream);
  if (e == cudaSuccess && T->gpart) e = cudaMemsetAsync(T->gpart, 0, 8 * (size_t)C->nx * sizeof(double), C->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaFree(h);
    return LBM_ECUDA;
  }
  int lin = 0;
  int st = LBM_OK;
  for (int sgi = T->nseg - 1; sgi >= 0 && st == LBM_OK; --sgi) {
    const int s0 = sgi * T->every, len = (sgi == T->nseg - 1) ? T->nsteps - s0 : T->every;
    // replay the segment: states s0 .. s0 + len - 1 into the segment buffer
    if (cudaMemcpyAsync(T->seg, T->ckpt[sgi], T->state_bytes, cudaMemcpyDeviceToDevice, C->stream) != cudaSuccess) {
      st = LBM_ECUDA;
      break;
    }
    if (C->stream && len == T->every) {
      const int l0 = lin;
      if (!T->bwd_graph[l0]) {
        st = capture(C, &T->bwd_graph[l0], &T->bwd_launches, [&]() {
          int l = l0;
          return segment_reverse<R>(C, T, len, &l);
        });
        if (st) break;
      }
      if (cudaGraphLaunch(T->bwd_graph[l0], C->stream) != cudaSuccess) {
        cudaGetLastError();
        st = LBM_ECUDA;
        break;
      }
      C->launches += T->bwd_launches;
      lin ^= len & 1;
    } else {
      st = segment_reverse<R>(C, T, len, &lin);
    }
  }
  if (st == LBM_OK) {
    // dL/dT: sum of the per-node parts in a fixed order; dL/dtheta; dL/df0
    e = lbm_reduce_rows(C, T->tacc, 0, C->ny, T->red, &C->launches);
    if (e == cudaSuccess && dl_dT)
      e = cudaMemcpyAsync(dl_dT, T->red, sizeof(double), cudaMemcpyDeviceToHost, C->stream);
    if (e == cudaSuccess && dl_dtheta)
      e = cudaMemcpyAsync(dl_dtheta, T->dtheta, 2 * (size_t)C->nx * sizeof(double), cudaMemcpyDeviceToHost,
                          C->stream);
    if (e == cudaSuccess && dl_df0) {
      double *tmp = nullptr;
      e = cudaMalloc(&tmp, 9 * n * sizeof(double));
      if (e == cudaSuccess) {
        k_to_double<R><<<(unsigned)((9 * n + B - 1) / B), B, 0, C->stream>>>((const R *)T->lam[lin], tmp, 9 * n);
        ++C->launches;
        e = cudaGetLastError();
        if (e == cudaSuccess)
          e = cudaMemcpyAsync(dl_df0, tmp, 9 * n * sizeof(double), cudaMemcpyDeviceToHost, C->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(C->stream);
        cudaFree(tmp);
      }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(C->stream);
    if (e != cudaSuccess) {
      cudaGetLastError();
      st = LBM_ECUDA;
    }
  }
  cudaStreamSynchronize(C->stream);
  cudaFree(h);
  return st;
}

}  // namespace

void lbm_adjoint_free_tape(lbm_ctx *C) {
  if (!C || !C->tape) return;
  lbm_tape *T = C->tape;
  cudaStreamSynchronize(C->stream);
  for (void *p : T->ckpt) cudaFree(p);
  cudaFree(T->seg);
  cudaFree(T->lam[0]);
  cudaFree(T->lam[1]);
  cudaFree(T->aux);
  cudaFree(T->rhob);
  cudaFree(T->tacc);
  cudaFree(T->gpart);
  cudaFree(T->dtheta);
  cudaFree(T->red);
  for (int p = 0; p < 2; ++p) {
    if (T->fwd_graph[p]) cudaGraphExecDestroy(T->fwd_graph[p]);
    if (T->bwd_graph[p]) cudaGraphExecDestroy(T->bwd_graph[p]);
  }
  cudaGetLastError();
  delete T;
  C->tape = nullptr;
}

extern "C" {

int lbm_adjoint_record(lbm_ctx *C, int nsteps, int checkpoint_every) {
  LbmRange nvtx_range("lbm_adjoint_record");
  if (!C || nsteps < 1 || checkpoint_every < 1) return LBM_EINVAL;
  if (C->status) return C->status;
  if (C->dp.n_iter > kMaxIter) return LBM_EUNSUPPORTED;
  lbm_adjoint_free_tape(C);
  lbm_tape *T = new (std::nothrow) lbm_tape();
  if (!T) return LBM_ENOMEM;
  C->tape = T;
  const size_t n = (size_t)C->nx * C->ny, rs = rsize(C);
  T->nsteps = nsteps;
  T->every = checkpoint_every < nsteps ? checkpoint_every : nsteps;
  T->nseg = (nsteps + T->every - 1) / T->every;
  T->state_bytes = 9 * n * rs;
  T->ckpt.assign(T->nseg, nullptr);
  bool ok = true;
  for (int k = 0; k < T->nseg && ok; ++k) ok = cudaMalloc(&T->ckpt[k], T->state_bytes) == cudaSuccess;
  ok = ok && cudaMalloc(&T->seg, (size_t)T->every * T->state_bytes) == cudaSuccess &&
       cudaMalloc(&T->lam[0], T->state_bytes) == cudaSuccess && cudaMalloc(&T->lam[1], T->state_bytes) == cudaSuccess &&
       cudaMalloc(&T->tacc, n * sizeof(double)) == cudaSuccess &&
       cudaMalloc(&T->dtheta, 2 * (size_t)C->nx * sizeof(double)) == cudaSuccess &&
       cudaMalloc(&T->red, sizeof(double)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    lbm_adjoint_free_tape(C);
    return LBM_ENOMEM;
  }
  // scratch of the FP64 reverse step's separate kernels
  if (C->precision == 64 &&
      (cudaMalloc(&T->aux, 5 * n * rs) != cudaSuccess || cudaMalloc(&T->rhob, n * rs) != cudaSuccess ||
       cudaMalloc(&T->gpart, 8 * (size_t)C->nx * sizeof(double)) != cudaSuccess ||
       (!C->d_fields && cudaMalloc(&C->d_fields, 3 * n * rs) != cudaSuccess))) {
    cudaGetLastError();
    lbm_adjoint_free_tape(C);
    return LBM_ENOMEM;
  }
  // run the steps, keeping the state at each segment start
  for (int sg = 0; sg < T->nseg; ++sg) {
    const int len = sg == T->nseg - 1 ? nsteps - sg * T->every : T->every;
    int st = LBM_OK;
    if (cudaMemcpyAsync(T->ckpt[sg], C->f[C->cur], T->state_bytes, cudaMemcpyDeviceToDevice, C->stream) !=
        cudaSuccess) {
      cudaGetLastError();
      st = LBM_ECUDA;
    }
    auto steps = [&](int count, int cur) {
      ACK(lbm_launch_steps(C, cur, count, &C->launches));
      return LBM_OK;
    };
    if (st == LBM_OK && C->stream && len == T->every) {
      const int p = C->cur;
      if (!T->fwd_graph[p]) st = capture(C, &T->fwd_graph[p], &T->fwd_launches, [&]() { return steps(len, p); });
      if (st == LBM_OK) {
        if (cudaGraphLaunch(T->fwd_graph[p], C->stream) != cudaSuccess) {
          cudaGetLastError();
          st = LBM_ECUDA;
        } else {
          C->launches += T->fwd_launches;
        }
      }
    } else if (st == LBM_OK) {
      st = steps(len, C->cur);
    }
    if (st) {
      lbm_adjoint_free_tape(C);
      C->status = st;
      return st;
    }
    C->cur ^= len & 1;
    C->steps += len;
  }
  if (cudaStreamSynchronize(C->stream) != cudaSuccess) {
    cudaGetLastError();
    lbm_adjoint_free_tape(C);
    return LBM_ECUDA;
  }
  return lbm_status(C);
}

int lbm_adjoint_backward(lbm_ctx *C, const double *dl_drho, double *dl_dtheta, double *dl_dT, double *dl_df0) {
  LbmRange nvtx_range("lbm_adjoint_backward");
  if (!C || !dl_drho) return LBM_EINVAL;
  if (!C->tape) return LBM_EINVAL;
  if (C->status == LBM_ECUDA) return C->status;
  return C->precision == 64 ? backward<double>(C, C->tape, dl_drho, dl_dtheta, dl_dT, dl_df0)
                            : backward<float>(C, C->tape, dl_drho, dl_dtheta, dl_dT, dl_df0);
}

int lbm_adjoint_release(lbm_ctx *C) {
  if (!C) return LBM_EINVAL;
  lbm_adjoint_free_tape(C);
  return LBM_OK;
}

}  // extern "C"
