// lbm_adjoint.cu -- discrete adjoint (reverse-time) of the canonical step.
//
// Forward step n -> n+1 (lbm_canon.cu): rho, psi, U (Eqs. 1, 10-11); ghost rows
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
#include "lbm_round.cuh"

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

using lbm_round::over;
using lbm_round::quot;
using lbm_round::vfma;

constexpr int kMaxIter = 64;

// Row k of M times v, left to right (the products by 2 and 4 are exact, so the
// fused ones round as separate ones).
template <typename R>
__device__ __forceinline__ R moment(int k, const R (&v)[9]) {
  R acc = (R)0;
  bool first = true;
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const R c = (R)MC(k, a);
    if (c == (R)0) continue;
    acc = first ? c * v[a] : (c == (R)1 ? acc + v[a] : (c == (R)-1 ? acc - v[a] : vfma(c, v[a], acc)));
    first = false;
  }
  return acc;
}

// psi_U with a shorter division by 3.
template <typename R>
__device__ __forceinline__ void node_eos(const Mdl<R> &m, R rho, R &psi, R &U) {
  U = pressure(m, rho) - over<3>(rho);
  psi = sqrt(fmax((R)0, (R)-2 * U));
}

template <typename R>
__device__ __forceinline__ void eos_derivs(const Mdl<R> &m, R rho, R &dp_drho, R &dp_dT) {
  if (m.kind == LBM_EOS_CARNAHAN_STARLING) {
    // p = rho R T Z(eta) - a rho^2, Z = N/D, N = 1 + eta + eta^2 - eta^3, D = (1 - eta)^3, eta = b rho/4:
    // dp/drho = R T (Z + eta dZ/deta) - 2 a rho,  dZ/deta = N'/D + 3 N/(1 - eta)^4
    R eta = (m.b * rho) * (R)0.25;
    R om = (R)1 - eta;
    R num = (((R)1 + eta) + eta * eta) - (eta * eta) * eta;
    R dnum = ((R)1 + (R)2 * eta) - (R)3 * (eta * eta);
    R den = (om * om) * om;
    const R y = (R)1 / den;
    R Z = quot(num, den, y);
    R dZ = quot(dnum, den, y) + ((R)3 * num) / (den * om);
    dp_drho = (m.Rg * m.T) * (Z + eta * dZ) - (R)2 * (m.a * rho);
    dp_dT = (rho * m.Rg) * Z;
  } else {
    dp_dT = (R)0;
    dp_drho = rho <= m.r1 ? m.thv : (rho <= m.r2 ? m.thm : m.thl);
  }
}

// Eq. 14's sums over the solid neighbours of a fluid node of row y.
template <typename R>
__device__ __forceinline__ void solid_sums(const Mdl<R> &m, int y, R &ssx, R &ssy) {
  ssx = ssy = (R)0;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const R ts = m.solid_row(m.wy(y + EY(a))) ? wgt<R>(a) : (R)0;
    if (EX(a)) ssx = EX(a) > 0 ? ssx + ts : ssx - ts;
    if (EY(a)) ssy = EY(a) > 0 ? ssy + ts : ssy - ts;
  }
}

// Eq. 9 force (+ Eq. 14) at a fluid node of row y; nb(ex, ey) is the index of a
// neighbour in psi and U.
template <typename R, typename Nb>
__device__ __forceinline__ void force(const Mdl<R> &m, const R *__restrict__ psi, const R *__restrict__ U, int y, Nb nb,
                                      R &Fx, R &Fy) {
  const R psi0 = psi[nb(0, 0)];
  R spx = (R)0, spy = (R)0, sUx = (R)0, sUy = (R)0;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const auto j = nb(EX(a), EY(a));
    const R tp = wgt<R>(a) * psi[j], tu = wgt<R>(a) * U[j];
    if (EX(a)) {
      spx = EX(a) > 0 ? spx + tp : spx - tp;
      sUx = EX(a) > 0 ? sUx + tu : sUx - tu;
    }
    if (EY(a)) {
      spy = EY(a) > 0 ? spy + tp : spy - tp;
      sUy = EY(a) > 0 ? sUy + tu : sUy - tu;
    }
  }
  const R cpsi = -(((R)1 - m.A) * psi0);
  Fx = -(m.A * sUx) - cpsi * spx;
  Fy = -(m.A * sUy) - cpsi * spy;
  if (m.wetting == LBM_WET_MARTYS_CHEN) {
    R ssx, ssy;
    solid_sums(m, y, ssx, ssy);
    const R gp = m.Gw * psi0;
    Fx = Fx - gp * ssx;
    Fy = Fy - gp * ssy;
  }
}

// Factors of the transposed collision that every node shares.
template <typename R>
struct AdjRates {
  R m[9], S[9];  // 1 - s_k, 1 - s_k/2
  explicit AdjRates(const lbm_dev_params &P) {
    for (int k = 0; k < 9; ++k) {
      m[k] = (R)1 - (R)P.s[k];
      S[k] = (R)1 - (R)0.5 * (R)P.s[k];
    }
  }
};

// Transpose of the collision at one fluid node: from ls = dL/df* (pulled back
// through the streaming), the populations f, rho and F to the part of dL/df that
// passes through the moments (cl), and aux = dL/d(Fx, Fy, Qxx, Qyy, Qxy).
template <typename R>
__device__ __forceinline__ void adj_collide(const Mdl<R> &m, const AdjRates<R> &K, const R (&f)[9], const R (&ls)[9],
                                            R rho, R Fx, R Fy, R (&cl)[9], R (&aux)[5]) {
  const R ir = (R)1 / rho;
  const R vx = quot(moment(3, f) + (R)0.5 * Fx, rho, ir), vy = quot(moment(5, f) + (R)0.5 * Fy, rho, ir);
  const R v2 = vx * vx + vy * vy;
  // f* = M^T diag(1/N) m*  ->  dL/dm*_k = sum_a M_ka ls_a / N_k
  const R msb[9] = {over<9>(moment(0, ls)),  over<36>(moment(1, ls)), over<36>(moment(2, ls)),
                    over<6>(moment(3, ls)),  over<12>(moment(4, ls)), over<6>(moment(5, ls)),
                    over<12>(moment(6, ls)), over<4>(moment(7, ls)),  over<4>(moment(8, ls))};
  R mb[9];
  // m*_k = m_k - s_k (m_k - meq_k) + (1 - s_k/2) S_k + C_k
  R meqb[9], Sb[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    mb[k] = K.m[k] * msb[k];
    meqb[k] = m.s[k] * msb[k];
    Sb[k] = K.S[k] * msb[k];
  }
  // C_1 = 1.5 s_1 (Qxx + Qyy), C_7 = -s_7 (Qxx - Qyy), C_8 = -s_8 Qxy
  aux[2] = ((R)1.5 * m.s[1]) * msb[1] - m.s[7] * msb[7];
  aux[3] = ((R)1.5 * m.s[1]) * msb[1] + m.s[7] * msb[7];
  aux[4] = -(m.s[8] * msb[8]);
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
  const R wx = quot(vxb, rho, ir), wy = quot(vyb, rho, ir);
  mb[3] = mb[3] + wx;
  mb[5] = mb[5] + wy;
  aux[0] = Fxb + (R)0.5 * wx;
  aux[1] = Fyb + (R)0.5 * wy;
  rhob = rhob - quot(vxb * vx + vyb * vy, rho, ir);
  // m = M f and rho = sum_a f_a
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    R acc = rhob;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const R c = (R)MC(k, a);
      if (c == (R)0) continue;
      acc = c == (R)1 ? acc + mb[k] : (c == (R)-1 ? acc - mb[k] : vfma(c, mb[k], acc));
    }
    cl[a] = acc;
  }
}

// dL/drho and dL/dT of node (row y) through psi and U, gathered from the aux of
// the fluid nodes whose stencils hold it; ax(ex, ey) is the index of a neighbour
// in the planes aux + k * an, nb(ex, ey) its index in psi.  rho: its density.
// aux is 0 at solid nodes (and psi finite), so that they add nothing.
template <typename R, typename Nb, typename Ax>
__device__ __forceinline__ void adj_psi(const Mdl<R> &m, const R *__restrict__ psi, const R *__restrict__ aux,
                                        size_t an, int y, R rho, Nb nb, Ax ax, R &rb, R &tb) {
  const R pre = m.kappa * (R)-0.5;
  const R omA = (R)1 - m.A;
  const R psi_p = psi[nb(0, 0)], Ap = m.A * psi_p;
  R pb = (R)0, ub = (R)0;
  // fluid nodes q = p - e_a hold p in their stencil in direction a:
  //   dF(q)/dpsi_p = (1-A) psi_q w_a e_a,  dF(q)/dU_p = -A w_a e_a,
  //   dQ_ij(q)/dpsi_p = pre w_a e_ai e_aj ((1-A) psi_q + A psi_p)
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const int ex = EX(a), ey = EY(a);
    const R *q = aux + ax(-ex, -ey);
    const R w = wgt<R>(a), c = omA * psi[nb(-ex, -ey)];
    R eF, eQ;
    if (ey == 0) {
      eF = ex > 0 ? q[0] : -q[0];
      eQ = q[2 * an];
    } else if (ex == 0) {
      eF = ey > 0 ? q[an] : -q[an];
      eQ = q[3 * an];
    } else {
      eF = (ex > 0 ? q[0] : -q[0]) + (ey > 0 ? q[an] : -q[an]);
      eQ = (q[2 * an] + q[3 * an]) + (ex * ey > 0 ? q[4 * an] : -q[4 * an]);
    }
    pb = pb + c * w * eF + pre * w * eQ * (c + Ap);
    ub = ub - m.A * w * eF;
  }
  // own terms: dF/dpsi_0 = (1-A) s_psi (+ Eq. 14), dQ_ii/dpsi_0 = pre ((1-A) q1_ii - psi_0),
  // dQ_xy/dpsi_0 = pre (1-A) q1_xy
  R spx = (R)0, spy = (R)0, qxx1 = (R)0, qyy1 = (R)0, qxy1 = (R)0;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const int ex = EX(a), ey = EY(a);
    const R w = wgt<R>(a), pn = psi[nb(ex, ey)], tp = w * pn, t1 = w * (pn - psi_p);
    if (ex) {
      spx = ex > 0 ? spx + tp : spx - tp;
      qxx1 = qxx1 + t1;
    }
    if (ey) {
      spy = ey > 0 ? spy + tp : spy - tp;
      qyy1 = qyy1 + t1;
    }
    if (ex && ey) qxy1 = ex * ey > 0 ? qxy1 + t1 : qxy1 - t1;
  }
  const R *o = aux + ax(0, 0);
  const R Fxb = o[0], Fyb = o[an];
  const bool fluid = !m.solid_row(y);
  pb = pb + omA * (Fxb * spx + Fyb * spy);
  if (m.wetting == LBM_WET_MARTYS_CHEN && fluid) {
    R ssx, ssy;
    solid_sums(m, y, ssx, ssy);
    pb = pb - m.Gw * (Fxb * ssx + Fyb * ssy);
  }
  pb = pb + pre * (omA * (o[2 * an] * qxx1 + o[3 * an] * qyy1 + o[4 * an] * qxy1) - psi_p * (o[2 * an] + o[3 * an]));
  // to dL/drho (and dL/dT) through U = p(rho) - rho/3 and psi = sqrt(-2U)
  rb = tb = (R)0;
  const bool ghost = !fluid && m.wetting == LBM_WET_GEOMETRIC;
  if (fluid || (ghost && rho < m.rho_max)) {
    R dp, dpT;
    eos_derivs(m, rho, dp, dpT);
    const R ut = ub - (psi_p > (R)0 ? pb / psi_p : (R)0);
    rb = ut * (dp - (R)1 / (R)3);
    tb = ut * dpT;
  }
}

// Transpose of the ghost rule at one wall node, from gb = dL/d(its density):
// part = dL/d(rho(x-1), rho(x+1), rho(x) of the boundary row, rho(x) of the
// second row); cb, cotb: dL/d(c, cot).  MAX: most iterations of Eq. 20.
template <int MAX, typename R>
__device__ __forceinline__ void adj_ghost(int n_iter, R ghost_max, R rim1, R ri1, R rip1, R ri2, R c, R cot, R gb, R (&part)[4],
                                          R &cb, R &cotb) {
  const R a = rip1 - rim1;
  // forward again, keeping the iterates: g_{k+1} = ri2 + c s_k, s_k = sqrt(a^2 + d_k^2), d_k = ri2 - g_k
  R d[MAX], sq[MAX];
  R g;
  if (n_iter <= 0) {
    g = ri2 + cot * fabs(a);
  } else {
    g = ri2;
    R dk = (R)2 * (ri2 - ri1);
#pragma unroll(MAX <= 4 ? MAX : 1)
    for (int k = 0; k < MAX; ++k) {
      if (k >= n_iter) break;
      d[k] = dk;
      sq[k] = sqrt(a * a + dk * dk);
      g = ri2 + c * sq[k];
      dk = ri2 - g;
    }
  }
  if (!(g > (R)0 && g < ghost_max)) gb = (R)0;  // clamped: no gradient
  R ab = (R)0, ri1b = (R)0, ri2b = (R)0;
  cb = cotb = (R)0;
  if (n_iter <= 0) {
    ri2b = gb;
    cotb = gb * fabs(a);
    ab = a > (R)0 ? gb * cot : (a < (R)0 ? -(gb * cot) : (R)0);
  } else {
    R gbar = gb;
#pragma unroll(MAX <= 4 ? MAX : 1)
    for (int k = MAX - 1; k >= 0; --k) {
      if (k >= n_iter) continue;
      ri2b = ri2b + gbar;
      cb = cb + gbar * sq[k];
      const R t = sq[k] > (R)0 ? (gbar * c) / sq[k] : (R)0;
      const R db = t * d[k];
      ab = ab + t * a;
      if (k >= 1) {  // d_k = ri2 - g_k
        ri2b = ri2b + db;
        gbar = -db;
      } else {  // d_0 = 2 (ri2 - ri1)
        ri2b = ri2b + (R)2 * db;
        ri1b = ri1b - (R)2 * db;
      }
    }
  }
  part[0] = -ab;
  part[1] = ab;
  part[2] = ri1b;
  part[3] = ri2b;
}
// the general count, out of the way of the code that runs
template <typename R>
__device__ __noinline__ void adj_ghost_any(int n_iter, R ghost_max, R rim1, R ri1, R rip1, R ri2, R c, R cot, R gb,
                                           R (&part)[4], R &cb, R &cotb) {
  adj_ghost<kMaxIter>(n_iter, ghost_max, rim1, ri1, rip1, ri2, c, cot, gb, part, cb, cotb);
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
// Small domains are bound by the latency of a kernel and by its one CTA per SM,
// whose 15 warps issue in 38% of the cycles (256 x 128, waiting for loads, fixed
// latencies, barriers and shared memory in equal parts): five kernels with four global round trips
// of fields, aux and dL/drho took longer than the repeated work at the tiles'
// edges (1.8 times the fields, 1.4 times the collisions), which at any size is
// also paid for by the 170 bytes a node that are not moved.  The arithmetic was
// then cut without a change of its bits (no products with the zeros of e and M,
// shared and constant divisors as in quot(), factors of the rates from the host),
// and what a thread adds to (tacc, dtheta) is loaded ahead.  Reverse step with
// its replay, us, five kernels -> one -> now: 256 x 128 21.9 -> 12.0 -> 9.9,
// 800 x 400 61 -> 55 -> 43, 1600 x 800 245 -> 238 -> 159.  In FP64 the repeated
// work costs more than it saves (the FP64 pipe is the limit: 800 x 400 816 us,
// in one kernel 1040), so FP64 keeps the kernels below: 682 now; 256 x 128
// 129 -> 111.
template <typename R>
__global__ void __launch_bounds__(kStepThreads)
    k_adj_step(Mdl<R> m, AdjRates<R> K, int strips, int bands, const R *__restrict__ f, const R *__restrict__ lam_in,
               R *__restrict__ lam_out, const double *__restrict__ coef, const double *__restrict__ dcoef,
               double *__restrict__ tacc, double *__restrict__ dtheta, int *flag) {
  constexpr int kAN = (kAH + 2) * kAW;  // aux: a row of zeros beyond each wall
  __shared__ R srho[kFH * kFW], spsi[kFH * kFW], sU[kFH * kFW];
  __shared__ R saux[5 * kAN];
  __shared__ R sgp[2][4][kAW];  // ghost-rule parts by wall, part, column (as in aux)
  const int band = (int)(blockIdx.x / (unsigned)strips);
  const int x0 = ((int)blockIdx.x - band * strips) * kTW, wr = min(kTW, m.nx - x0);
  const int first = m.walls ? 1 : 0, rows = m.walls ? m.ny - 2 : m.ny;
  // equal bands: with walls the outer ones hold both rows that a ghost node reads
  const int ya = first + (int)((long long)band * rows / bands), yb = first + (int)((long long)(band + 1) * rows / bands);
  const int hr = yb - ya;
  const size_t n = (size_t)m.nx * m.ny;
  const bool geo = m.walls && m.wetting == LBM_WET_GEOMETRIC;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // this thread's node: rows ya - 1 .. yb, columns x0 - 2 .. x0 + wr + 1
  const int cy = threadIdx.x / kAW, cx = threadIdx.x - cy * kAW, v = ya - 1 + cy;
  const bool on = cy < hr + 2 && cx < wr + 4;  // (in a walled domain all these rows exist)
  const int y = m.wy(v), x = m.wx(x0 - 2 + cx), w = y == 0 ? 0 : 1;
  const bool solid = m.solid_row(y), own = on && cx >= 2 && cx < wr + 2 && (solid || (cy >= 1 && cy <= hr));
  const bool wall = on && solid && geo && cx >= 1 && cx < wr + 3;  // a ghost node whose transposed rule is needed
  const size_t i = (size_t)y * m.nx + x;
  const int jf = (cy + 1) * kFW + cx + 1, ja = (cy + 1) * kAW + cx;  // its place among the fields and aux
  auto nb = [&](int ex, int ey) { return jf + ey * kFW + ex; };
  auto ax = [&](int ex, int ey) { return ja + ey * kAW + ex; };
  R c = (R)0, cot = (R)0;
  double dc = 0.0, dcot = 0.0;
  if (wall) {
    c = (R)coef[w * m.nx + x];
    cot = (R)coef[2 * m.nx + w * m.nx + x];
    dc = dcoef[w * m.nx + x];
    dcot = dcoef[2 * m.nx + w * m.nx + x];
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  R ls[9], fl[9], cl[9];
  if (on && !solid) {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int yt = m.wy(y + EY(a));
      ls[a] = m.solid_row(yt) ? lam_in[OPP(a) * n + i] : lam_in[a * n + (size_t)yt * m.nx + m.wx(x + EX(a))];
      fl[a] = f[a * n + i];
    }
  }
  // the sums this thread adds to, loaded ahead of their use
  const double t0 = own ? tacc[i] : 0.0, th0 = own && wall ? dtheta[w * m.nx + x] : 0.0;
  // fields: rows ya - 2 .. yb + 1, columns x0 - 3 .. x0 + wr + 2
  bool bad = false;
  const int t = threadIdx.x, fy = t / kFW, fx = t - fy * kFW, fv = ya - 2 + fy;
  if (fy < hr + 4 && fx < wr + 6) {
    R r = (R)0, psi = (R)0, U = (R)0;
    if (!(m.walls && (fv < 0 || fv >= m.ny))) {
      const int y = m.wy(fv), x = m.wx(x0 - 3 + fx);
      if (!m.solid_row(y)) {
        r = node_rho(f, n, (size_t)y * m.nx + x);
        node_eos(m, r, psi, U);
        bad |= !(r > (R)0) || r > m.rho_max;
      } else if (geo) {
        const int w = y == 0 ? 0 : 1;
        const size_t b1 = (size_t)(w == 0 ? 1 : m.ny - 2) * m.nx, b2 = (size_t)(w == 0 ? 2 : m.ny - 3) * m.nx;
        r = ghost_rho(m, node_rho(f, n, b1 + m.wx(x - 1)), node_rho(f, n, b1 + x), node_rho(f, n, b1 + m.wx(x + 1)),
                      node_rho(f, n, b2 + x), (R)coef[w * m.nx + x], (R)coef[2 * m.nx + w * m.nx + x]);
        if (r < m.rho_max) node_eos(m, r, psi, U);
      }
    }
    srho[t] = r;
    spsi[t] = psi;
    sU[t] = U;
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
  if (on) {
    R a5[5] = {(R)0, (R)0, (R)0, (R)0, (R)0};
    if (!solid) {
      R Fx, Fy;
      force(m, spsi, sU, y, nb, Fx, Fy);
      adj_collide(m, K, fl, ls, srho[jf], Fx, Fy, cl, a5);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      saux[k * kAN + ja] = a5[k];
      if (solid) saux[k * kAN + ja + (cy == 0 ? -kAW : kAW)] = (R)0;
    }
  }
  __syncthreads();
  // dL/drho: the tile's nodes, and the ghost nodes of one more column each side
  R rb = (R)0;
  if (own || wall) {
    R tb;
    adj_psi(m, spsi, saux, kAN, y, srho[jf], nb, ax, rb, tb);
    if (own) tacc[i] = t0 + (double)tb;
    if (wall) {
      const int s = w == 0 ? kFW : -kFW;
      R part[4], cb, cotb;
      if (m.n_iter <= 4)
        adj_ghost<4>(m.n_iter, m.ghost_max, srho[jf + s - 1], srho[jf + s], srho[jf + s + 1], srho[jf + 2 * s], c, cot, rb, part, cb, cotb);
      else
        adj_ghost_any(m.n_iter, m.ghost_max, srho[jf + s - 1], srho[jf + s], srho[jf + s + 1], srho[jf + 2 * s], c, cot, rb, part, cb,
                      cotb);
      if (own) dtheta[w * m.nx + x] = th0 + (m.n_iter > 0 ? (double)cb * dc : (double)cotb * dcot);
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
      if (y == y1) r += (double)sgp[w][0][cx + 1] + (double)sgp[w][1][cx - 1] + (double)sgp[w][2][cx];
      if (y == y2) r += (double)sgp[w][3][cx];
    }
    rb = (R)r;
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) lam_out[a * n + i] = cl[a] + rb;
}

// ---- the four kernels of a reverse step on whole fields (FP64, see reverse_step) --

template <typename R>
__global__ void k_adj_collide(Mdl<R> m, AdjRates<R> K, const R *__restrict__ f, const R *__restrict__ fields,
                              const R *__restrict__ lam_in, R *__restrict__ lam_out, R *__restrict__ aux) {
  size_t n = (size_t)m.nx * m.ny;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int y = (int)(i / m.nx), x = (int)(i - (size_t)y * m.nx);
  if (m.solid_row(y)) {
#pragma unroll
    for (int k = 0; k < 5; ++k) aux[k * n + i] = (R)0;
    return;
  }
  // adjoint of the post-collision populations (transpose of the push streaming)
  R ls[9], fl[9], cl[9], ax[5];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    int yt = m.wy(y + EY(a));
    ls[a] = m.solid_row(yt) ? lam_in[OPP(a) * n + i] : lam_in[a * n + (size_t)yt * m.nx + m.wx(x + EX(a))];
    fl[a] = f[a * n + i];
  }
  R Fx, Fy;
  force(m, fields + n, fields + 2 * n, y, FieldNb<R>{m, y, x}, Fx, Fy);
  adj_collide(m, K, fl, ls, fields[i], Fx, Fy, cl, ax);
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
  R rb, tb;
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
  R part[4], cb, cotb;
  const R c = (R)coef[w * m.nx + x], cot = (R)coef[2 * m.nx + w * m.nx + x], gb = rhob[(size_t)yg * m.nx + x];
  if (m.n_iter <= 4)
    adj_ghost<4>(m.n_iter, m.ghost_max, r1[m.wx(x - 1)], r1[x], r1[m.wx(x + 1)], r2[x], c, cot, gb, part, cb, cotb);
  else
    adj_ghost_any(m.n_iter, m.ghost_max, r1[m.wx(x - 1)], r1[x], r1[m.wx(x + 1)], r2[x], c, cot, gb, part, cb, cotb);
  dtheta[w * m.nx + x] +=
      m.n_iter > 0 ? (double)cb * dcoef[w * m.nx + x] : (double)cotb * dcoef[2 * m.nx + w * m.nx + x];
#pragma unroll
  for (int k = 0; k < 4; ++k) gpart[((size_t)w * 4 + k) * m.nx + x] = (double)part[k];
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
    ACK(cudaLaunchKernelEx(&cfg, k_adj_step<R>, m, AdjRates<R>(C->dp), strips, bands, (const R *)f, (const R *)lam_in, lam_out,
                           (const double *)C->d_coef, (const double *)C->d_dcoef, T->tacc, T->dtheta, C->d_flag));
    ++C->launches;
    return LBM_OK;
  } else {
    const int B = 256;
    const size_t n = (size_t)C->nx * C->ny;
    const unsigned g = (unsigned)((n + B - 1) / B), gw = (unsigned)((2 * C->nx + B - 1) / B);
    const R *fields = (const R *)C->d_fields;
    ACK(lbm_ref_fields(C, (const double *)f, (double *)C->d_fields, &C->launches));
    k_adj_collide<R><<<g, B, 0, C->stream>>>(m, AdjRates<R>(C->dp), (const R *)f, fields, lam_in, lam_out, (R *)T->aux);
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
