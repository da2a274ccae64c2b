// lbm_canon.cu -- the step in the canonical evaluation order (the oracle's: the
// equations term by term, sums left to right, no contraction), one kernel per
// step: FP64 domains, and FP32 domains whose width the fused kernels do not take.
// Every result has the bits of that plain form; the operations that cost most are
// only arranged anew:
//  - a product by a power of two is exact, so the sum it goes into takes it as
//    a fused multiply-add with the same single rounding, and such factors move
//    freely through roundings (4 f_0 - 2 f_1 is twice 2 f_0 - f_1);
//  - x / 3, x / 9, x / 36, x / 6, x / 12: one product and one fused
//    multiply-add (div_const) instead of a general division;
//  - other FP32 quotients and square roots are corrected approximations, packed
//    (quotients and root0_in_range, lbm_round.cuh);
//  - values that several sums use in the same order are formed once (prefixes
//    of the inverse transform, psi^2, and, per node instead of per neighbour,
//    the weighted psi and U of the FP64 kernel).
// About 350 FP64 operations per node instead of 700, and one pass over the
// populations instead of two and a pass over three fields (FP32: 72 bytes per
// node instead of 132).  us per step, before -> now: FP64 100 x 60 29.6 -> 16.7,
// 400 x 200 104 -> 80; FP32 1001 x 501 30.4 -> 11.4, 2047 x 1025 131 -> 44.
// FP64 is bound by the FP64 pipe (0.5 lanes per clock and SM quarter): 55% of its
// cycles at 400 x 200, and at 100 x 60 one warp's chain through it (25%, 2.8 warps on
// an SM).  FP32 waits for its loads at 28 warps per SM, of which 60% of the cycles
// issue an instruction (1001 x 501; 14% of DRAM throughput).
#include <math.h>
#include <string.h>

#include <type_traits>

#include "lbm_internal.h"
#include "lbm_round.cuh"

namespace {

using namespace lbm_round;

// a where x <= lim, else b
__device__ __forceinline__ F2 where_le(F2 x, float lim, F2 a, F2 b) {
  return {make_float2(x.v.x <= lim ? a.v.x : b.v.x, x.v.y <= lim ? a.v.y : b.v.y)};
}
template <class R>
__device__ __forceinline__ R where_le(R x, R lim, R a, R b) {
  return x <= lim ? a : b;
}

// Model constants, evaluated on the host in the kernel's precision in the order
// in which the plain form evaluates them.
template <class R>
struct Canon {
  int nx, ny, walls, kind, n_iter, wetting;
  int strips, sw;                         // strips of sw columns
  R b4, Rg, T, a;                         // Carnahan-Starling (b/4)
  R thv, thm, thl, r1, r2, p1, p2;        // Eq. 11; its pressure at r1 and at r2
  R A, omA, c2, pre, Gw, ss_dn, ss_up;    // 1 - A, A/2, -kappa/2, sum_a w_a S e_ay at the two walls
  R s1, s2, s3, s4, s7, h1, h2, h3, h4, h7, h7x2, c15;  // rates, 1 - s/2, 2 (1 - s_7/2), 1.5 s_1
  R rho_max, ghost_max;
  R z3h, z3l, z9h, z9l, z36h, z36l, z6h, z6l, z12h, z12l;  // 1/d as a sum of two numbers
  unsigned plain_lo, plain_len;           // bits of the densities [lo, hi] of plain(), hi - lo

  explicit Canon(const lbm_ctx *C) {
    const lbm_dev_params &P = C->dp;
    nx = P.nx, ny = P.ny, walls = P.walls, kind = P.eos_kind, n_iter = P.n_iter, wetting = P.wetting;
    strips = sw = 0;
    b4 = (R)P.b * (R)0.25, Rg = (R)P.R, T = (R)P.T, a = (R)P.a;
    thv = (R)P.thv, thm = (R)P.thm, thl = (R)P.thl, r1 = (R)P.r1, r2 = (R)P.r2;
    p1 = r1 * thv;
    const R dp = (r2 - r1) * thm;
    p2 = p1 + dp;
    A = (R)P.A, omA = (R)1 - A, c2 = A * (R)0.5, pre = (R)P.kappa * ((R)-1 * (R)0.5), Gw = (R)P.Gw;
    const R w1 = (R)1 / (R)3, w2 = (R)1 / (R)12;
    ss_up = (w1 + w2) + w2;
    ss_dn = -ss_up;
    s1 = (R)P.s[1], s2 = (R)P.s[2], s3 = (R)P.s[3], s4 = (R)P.s[4], s7 = (R)P.s[7];
    auto half = [](R s) {
      const R t = (R)0.5 * s;
      return (R)1 - t;
    };
    h1 = half(s1), h2 = half(s2), h3 = half(s3), h4 = half(s4), h7 = half(s7), h7x2 = (R)2 * h7, c15 = (R)1.5 * s1;
    rho_max = (R)P.rho_max, ghost_max = (R)P.ghost_max;
    const_reciprocal((R)3, &z3h, &z3l);
    const_reciprocal((R)9, &z9h, &z9l);
    const_reciprocal((R)36, &z36h, &z36l);
    const_reciprocal((R)6, &z6h, &z6l);
    const_reciprocal((R)12, &z12h, &z12l);
    // Densities whose quotients and square root stay where lbm_round.cuh takes the
    // corrected approximations: rho itself in [2^-40, 2^30]; for Carnahan-Starling
    // (1 - eta)^3 >= 2^-24, the numerator in [2^-80, 2^14] and the parts of U below
    // 2^38, for Eq. 11 U below 2^38.  U = p - rho/3, where p and rho/3 cancel, is a
    // multiple of their last place, 2^-66 or more, or 0.
    double lo = 0x1p-40, hi = 0x1p30;
    if (kind == LBM_EOS_CARNAHAN_STARLING) {
      lo = fmax(lo, 0x1p-78 / (P.R * P.T));
      hi = fmin(fmin(hi, (1.0 - 0x1p-7) * 4.0 / P.b), fmin(0x1p12 / (P.R * P.T), sqrt(0x1p36 / P.a)));
    } else {
      hi = fmin(hi, 0x1p34 / fmax(1.0, fmax(fmax(fabs(P.thv), fabs(P.thm)), fabs(P.thl))));
    }
    const float l = (float)lo, h = (float)hi;
    unsigned hb;
    memcpy(&plain_lo, &l, sizeof(l));
    memcpy(&hb, &h, sizeof(h));
    plain_len = hb - plain_lo;
    if (!(l < h)) plain_lo = 0x7fffffffu, plain_len = 0u;  // none (the bits of a NaN)
  }
};

// Both lanes of rho lie in [lo, hi]: positive numbers order like their bits.
__device__ __forceinline__ bool plain(const Canon<float> &m, F2 rho) {
  return __float_as_uint(rho.v.x) - m.plain_lo <= m.plain_len && __float_as_uint(rho.v.y) - m.plain_lo <= m.plain_len;
}
template <class R>
__device__ __forceinline__ bool plain(const Canon<R> &, R) {
  return true;
}

// psi and U of Eqs. 10-11; over(a, b) is a / b and root(a) is sqrt(max(0, a)).
template <class V, class R, class Over, class Root>
__device__ __forceinline__ void psi_U(const Canon<R> &m, V rho, V &psi, V &U, Over over, Root root) {
  auto bc = [](R c) { return Val<V>::bc(c); };
  V p;
  if (m.kind == LBM_EOS_CARNAHAN_STARLING) {
    const V eta = bc(m.b4) * rho, e2 = eta * eta, one = bc((R)1), om = one - eta;
    const V num = ((one + eta) + e2) - e2 * eta, den = (om * om) * om;
    p = over(((rho * bc(m.Rg)) * bc(m.T)) * num, den) - (bc(m.a) * rho) * rho;
  } else {
    p = where_le(rho, m.r1, rho * bc(m.thv),
                 where_le(rho, m.r2, bc(m.p1) + (rho - bc(m.r1)) * bc(m.thm),
                          bc(m.p2) + (rho - bc(m.r2)) * bc(m.thl)));
  }
  U = p - div_const(rho, m.z3h, m.z3l);
  psi = root(bc((R)-2) * U);
}
template <class V, class R>
__device__ __forceinline__ void psi_U(const Canon<R> &m, V rho, V &psi, V &U) {
  psi_U(m, rho, psi, U, [](V a, V b) { return a / b; }, [](V a) { return root0(a); });
}
// The same for a rho that is plain(m, rho).
__device__ __forceinline__ void psi_U_plain(const Canon<float> &m, F2 rho, F2 &psi, F2 &U) {
  psi_U(m, rho, psi, U, [](F2 a, F2 b) { return Reciprocal(b).under(a); }, [](F2 a) { return root0_in_range(a); });
}
__device__ __forceinline__ void psi_U_plain(const Canon<double> &m, double rho, double &psi, double &U) {
  psi_U(m, rho, psi, U);
}

// Ghost density, psi and U (Eqs. 19-21) from the densities around column x.
template <class R>
__device__ __forceinline__ void ghost(const Canon<R> &m, R rim1, R ri1, R rip1, R ri2, R c, R &g, R &psi, R &U) {
  const R a = rip1 - rim1;
  g = ri2;
  if (m.n_iter <= 0) {
    g = ri2 + c * fabs(a);
  } else {
    const R aa = a * a;
    R d = (R)2 * (ri2 - ri1);
    for (int k = 0; k < m.n_iter; ++k) {
      g = ri2 + c * sqrt(aa + d * d);
      d = ri2 - g;
    }
  }
  g = fmin(fmax(g, (R)0), m.ghost_max);
  psi = U = (R)0;
  if (g < m.rho_max) psi_U(m, g, psi, U);
}

// The neighbour values of a window: psi, psi^2, w psi, w U.
template <class V>
struct Nb {
  V p, p2, tp, tu;
};

constexpr int kH = 32;       // lanes of a row; a lane pair is columns t, t + 32
constexpr int kWP = kH + 4;  // window entries -2 .. kH + 1 at index i + 2

template <class V, int R>
struct Window;
template <int R>
struct Window<F2, R> {
  F2 p[R + 2][kWP], u[R + 2][kWP];
  __device__ __forceinline__ void put1(int row, int i, int lane, float psi, float U) {
    Val<F2>::set(p[row][i], lane, psi);
    Val<F2>::set(u[row][i], lane, U);
  }
  __device__ __forceinline__ void put(int row, int c, float psi, float U) {
    if (c <= kH + 1) put1(row, c + 2, 0, psi, U);
    if (c >= kH - 2) put1(row, c - kH + 2, 1, psi, U);
  }
  template <bool DIAG>
  __device__ __forceinline__ Nb<F2> at(int row, int i) const {
    const F2 w = Val<F2>::bc(DIAG ? 1.0f / 12.0f : 1.0f / 3.0f), a = p[row][i];
    return {a, a * a, w * a, w * u[row][i]};
  }
};
template <int R>
struct Window<double, R> {
  double p[R + 2][kWP], u[R + 2][kWP], p2[R + 2][kWP], p1w[R + 2][kWP], p2w[R + 2][kWP], u1w[R + 2][kWP],
      u2w[R + 2][kWP];
  __device__ __forceinline__ void put(int row, int c, double psi, double U) {
    const int i = c + 2;
    p[row][i] = psi;
    u[row][i] = U;
    p2[row][i] = psi * psi;
    p1w[row][i] = (1.0 / 3.0) * psi;
    p2w[row][i] = (1.0 / 12.0) * psi;
    u1w[row][i] = (1.0 / 3.0) * U;
    u2w[row][i] = (1.0 / 12.0) * U;
  }
  template <bool DIAG>
  __device__ __forceinline__ Nb<double> at(int row, int i) const {
    return {p[row][i], p2[row][i], DIAG ? p2w[row][i] : p1w[row][i], DIAG ? u2w[row][i] : u1w[row][i]};
  }
};

// Force (Eq. 9, + Eq. 14 with ss = sum_a w_a S e_ay) and Eq. 17 tensor of the
// node(s) at window row `row`, entry i.
template <class V, class R, class W>
__device__ __forceinline__ void force(const Canon<R> &m, const W &win, int row, int i, R ss, V &Fx, V &Fy, V &Qxx,
                                      V &Qyy, V &Qxy) {
  auto bc = [](R c) { return Val<V>::bc(c); };
  const V w1 = bc((R)1 / (R)3), w2 = bc((R)1 / (R)12);
  const Nb<V> n0 = win.template at<false>(row, i);
  V spx, spy, sUx, sUy, xx1, yy1, xy1, xx2, yy2, xy2;
  auto t1 = [&](const Nb<V> &n, V w) { return w * (n.p - n0.p); };
  auto t2 = [&](const Nb<V> &n, V w) { return w * (n.p2 - n0.p2); };
  Nb<V> n = win.template at<false>(row, i + 1);  // e1
  spx = n.tp, sUx = n.tu, xx1 = t1(n, w1), xx2 = t2(n, w1);
  n = win.template at<false>(row + 1, i);  // e2
  spy = n.tp, sUy = n.tu, yy1 = t1(n, w1), yy2 = t2(n, w1);
  n = win.template at<false>(row, i - 1);  // e3
  spx = spx - n.tp, sUx = sUx - n.tu, xx1 = xx1 + t1(n, w1), xx2 = xx2 + t2(n, w1);
  n = win.template at<false>(row - 1, i);  // e4
  spy = spy - n.tp, sUy = sUy - n.tu, yy1 = yy1 + t1(n, w1), yy2 = yy2 + t2(n, w1);
  n = win.template at<true>(row + 1, i + 1);  // e5
  V a = t1(n, w2), b = t2(n, w2);
  spx = spx + n.tp, sUx = sUx + n.tu, spy = spy + n.tp, sUy = sUy + n.tu;
  xx1 = xx1 + a, xx2 = xx2 + b, yy1 = yy1 + a, yy2 = yy2 + b, xy1 = a, xy2 = b;
  n = win.template at<true>(row + 1, i - 1);  // e6
  a = t1(n, w2), b = t2(n, w2);
  spx = spx - n.tp, sUx = sUx - n.tu, spy = spy + n.tp, sUy = sUy + n.tu;
  xx1 = xx1 + a, xx2 = xx2 + b, yy1 = yy1 + a, yy2 = yy2 + b, xy1 = xy1 - a, xy2 = xy2 - b;
  n = win.template at<true>(row - 1, i - 1);  // e7
  a = t1(n, w2), b = t2(n, w2);
  spx = spx - n.tp, sUx = sUx - n.tu, spy = spy - n.tp, sUy = sUy - n.tu;
  xx1 = xx1 + a, xx2 = xx2 + b, yy1 = yy1 + a, yy2 = yy2 + b, xy1 = xy1 + a, xy2 = xy2 + b;
  n = win.template at<true>(row - 1, i + 1);  // e8
  a = t1(n, w2), b = t2(n, w2);
  spx = spx + n.tp, sUx = sUx + n.tu, spy = spy - n.tp, sUy = sUy - n.tu;
  xx1 = xx1 + a, xx2 = xx2 + b, yy1 = yy1 + a, yy2 = yy2 + b, xy1 = xy1 - a, xy2 = xy2 - b;
  const V c1 = bc(m.omA) * n0.p, c2 = bc(m.c2), pre = bc(m.pre);
  Fx = c1 * spx - bc(m.A) * sUx;
  Fy = c1 * spy - bc(m.A) * sUy;
  if (m.wetting == LBM_WET_MARTYS_CHEN) Fy = Fy - (bc(m.Gw) * n0.p) * bc(ss);
  Qxx = pre * (c1 * xx1 + c2 * xx2);
  Qyy = pre * (c1 * yy1 + c2 * yy2);
  Qxy = pre * (c1 * xy1 + c2 * xy2);
}

// Momenta j_x, j_y, left to right in f_0 .. f_8 (also the first terms of q_x, q_y).
template <class V>
__device__ __forceinline__ void momentum(const V (&f)[9], V &d13, V &d24, V &jx, V &jy) {
  d13 = f[1] - f[3];
  d24 = f[2] - f[4];
  jx = (((d13 + f[5]) - f[6]) - f[7]) + f[8];
  jy = (((d24 + f[5]) + f[6]) - f[7]) - f[8];
}

// MRT collision of the node(s) at window row `row`, entry i; f: populations,
// rho: density, fs: post-collision populations.
template <class V, class R, class W>
__device__ __forceinline__ void collide(const Canon<R> &m, const W &win, int row, int i, const V (&f)[9], V rho,
                                        bool ok, R ss, V (&fs)[9]) {
  auto bc = [](R c) { return Val<V>::bc(c); };
  V Fx, Fy, Qxx, Qyy, Qxy, d13, d24, jx, jy;
  force(m, win, row, i, ss, Fx, Fy, Qxx, Qyy, Qxy);
  momentum(f, d13, d24, jx, jy);
  const V half = bc((R)0.5), two = bc((R)2), m2 = bc((R)-2), four = bc((R)4), m4 = bc((R)-4), quarter = bc((R)0.25);
  // moments (rho is the first), left to right in f_0 .. f_8
  V me = vfma(m4, f[0], -f[1]);
  me = ((me - f[2]) - f[3]) - f[4];
  me = vfma(two, f[8], vfma(two, f[7], vfma(two, f[6], vfma(two, f[5], me))));
  V mp = ((vfma(two, f[0], -f[1]) - f[2]) - f[3]) - f[4];  // half of 4 f_0 - 2 f_1 - ...
  mp = ((vfma(two, mp, f[5]) + f[6]) + f[7]) + f[8];
  const V qx = ((vfma(m2, d13, f[5]) - f[6]) - f[7]) + f[8];
  const V qy = ((vfma(m2, d24, f[5]) + f[6]) - f[7]) - f[8];
  const V nn = ((f[1] - f[2]) + f[3]) - f[4];
  const V no = ((f[5] - f[6]) + f[7]) - f[8];
  V vx, vy;
  quotients(vfma(half, Fx, jx), vfma(half, Fy, jy), rho, ok, vx, vy);
  const V vx2 = vx * vx, vy2 = vy * vy, v3 = bc((R)3) * (vx2 + vy2);
  const V vxF = vx * Fx, vyF = vy * Fy, S1 = bc((R)6) * (vxF + vyF);
  const V rvx = rho * vx, rvy = rho * vy;
  // m - s (m - meq) + (1 - s/2) S + C, divided by N
  V r0 = div_const(rho, m.z9h, m.z9l);
  V r1 = ((me - bc(m.s1) * (me - rho * (v3 - two))) + bc(m.h1) * S1) + bc(m.c15) * (Qxx + Qyy);
  V r2 = (mp - bc(m.s2) * (mp - rho * (bc((R)1) - v3))) - bc(m.h2) * S1;
  V r3 = (jx - bc(m.s3) * (jx - rvx)) + bc(m.h3) * Fx;
  V r4 = (qx - bc(m.s4) * (qx + rvx)) - bc(m.h4) * Fx;
  V r5 = (jy - bc(m.s3) * (jy - rvy)) + bc(m.h3) * Fy;
  V r6 = (qy - bc(m.s4) * (qy + rvy)) - bc(m.h4) * Fy;
  V r7 = ((nn - bc(m.s7) * (nn - rho * (vx2 - vy2))) + bc(m.h7x2) * (vxF - vyF)) - bc(m.s7) * (Qxx - Qyy);
  V r8 = ((no - bc(m.s7) * (no - rho * (vx * vy))) + bc(m.h7) * (vx * Fy + vy * Fx)) - bc(m.s7) * Qxy;
  r1 = div_const(r1, m.z36h, m.z36l);
  r2 = div_const(r2, m.z36h, m.z36l);
  r3 = div_const(r3, m.z6h, m.z6l);
  r4 = div_const(r4, m.z12h, m.z12l);
  r5 = div_const(r5, m.z6h, m.z6l);
  r6 = div_const(r6, m.z12h, m.z12l);
  // f* = M^T r; r7 and r8 still carry their factor 4
  const V mq = bc((R)-0.25);
  fs[0] = vfma(four, r2, vfma(m4, r1, r0));
  const V ax = vfma(m2, r2, r0 - r1);
  fs[1] = vfma(quarter, r7, vfma(m2, r4, ax + r3));
  fs[2] = vfma(mq, r7, vfma(m2, r6, ax + r5));
  fs[3] = vfma(quarter, r7, vfma(two, r4, ax - r3));
  fs[4] = vfma(mq, r7, vfma(two, r6, ax - r5));
  const V dg = vfma(two, r1, r0) + r2, dp = (dg + r3) + r4, dm = (dg - r3) - r4;
  fs[5] = vfma(quarter, r8, (dp + r5) + r6);
  fs[6] = vfma(mq, r8, (dm + r5) + r6);
  fs[7] = vfma(quarter, r8, (dm - r5) - r6);
  fs[8] = vfma(mq, r8, (dp - r5) - r6);
}

// Outputs of the kernel below: Step writes the state after the step, Speed the largest |u|^2 (as the bits
// of a non-negative double, which order like the number), Fields the fields.
template <class R>
struct Step {
  R *f;
};
struct Speed {
  unsigned long long *max2;
};
struct Fields {
  double *o[10];  // rho, psi, U, ux, uy, Fx, Fy, Qxx, Qyy, Qxy; NULL where not wanted
};

// What a CTA does with its window, per output.
template <class V, int R, class real>
__device__ __forceinline__ void emit(const Canon<real> &m, const Step<real> &out, const Window<V, R> &win,
                                     const real (&)[R + 2][Val<V>::N * kH + 4], int w, int lane, int, int y, int x0,
                                     const bool (&act)[Val<V>::N], bool node, bool, real ss, const V (&f)[9], V r, bool ok) {
  constexpr int N = Val<V>::N;
  if (!node) return;
  const size_t n = (size_t)m.nx * m.ny;
  const bool dn = m.walls && y == 1, up = m.walls && y == m.ny - 2;
  V fs[9];
  collide(m, win, w, lane + 2, f, r, ok, ss, fs);
  // streaming with half-way bounce-back
  const size_t ry = (size_t)y * m.nx, rd = (size_t)(y == 0 ? m.ny - 1 : y - 1) * m.nx,
               ru = (size_t)(y == m.ny - 1 ? 0 : y + 1) * m.nx;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (!act[j]) break;
    const int x = x0 + lane + j * kH, xm = x == 0 ? m.nx - 1 : x - 1, xp = x == m.nx - 1 ? 0 : x + 1;
    auto g = [&](int a) { return Val<V>::lane(fs[a], j); };
    real *const o = out.f;
    o[ry + x] = g(0);
    o[n + ry + xp] = g(1);
    o[3 * n + ry + xm] = g(3);
    o[(up ? 4 * n + ry : 2 * n + ru) + x] = g(2);
    o[up ? 7 * n + ry + x : 5 * n + ru + xp] = g(5);
    o[up ? 8 * n + ry + x : 6 * n + ru + xm] = g(6);
    o[(dn ? 2 * n + ry : 4 * n + rd) + x] = g(4);
    o[dn ? 5 * n + ry + x : 7 * n + rd + xm] = g(7);
    o[dn ? 6 * n + ry + x : 8 * n + rd + xp] = g(8);
  }
}

// |u|^2 in double of the velocity in the kernel's precision, as lbm_get_u gives
// it; its largest value, the square root of which is the largest |u| (both are
// monotone).  FP32: only nodes near the largest of their warp in single
// precision go through the FP64 pipe.
template <class V, int R, class real>
__device__ __forceinline__ void emit(const Canon<real> &m, const Speed &out, const Window<V, R> &win,
                                     const real (&)[R + 2][Val<V>::N * kH + 4], int w, int lane, int, int, int,
                                     const bool (&act)[Val<V>::N], bool node, bool, real ss, const V (&f)[9], V r, bool) {
  constexpr int N = Val<V>::N;
  V Fx, Fy, Qxx, Qyy, Qxy, d13, d24, jx, jy;
  if (node) {
    force(m, win, w, lane + 2, ss, Fx, Fy, Qxx, Qyy, Qxy);
    momentum(f, d13, d24, jx, jy);
    const V half = Val<V>::bc((real)0.5);
    Fx = vfma(half, Fx, jx) / r;
    Fy = vfma(half, Fy, jy) / r;
  }
  float near[N], top = 0.0f;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const float ux = node && act[j] ? (float)Val<V>::lane(Fx, j) : 0.0f;
    const float uy = node && act[j] ? (float)Val<V>::lane(Fy, j) : 0.0f;
    near[j] = ux * ux + uy * uy;
    top = fmaxf(top, near[j]);  // (NaN counts for nothing)
  }
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  const float lim = top > 1e-30f ? top * 0.99999f : 0.0f;  // (below, squares lose their precision)
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (node && act[j] && near[j] >= lim) {
      const double ux = (double)Val<V>::lane(Fx, j), uy = (double)Val<V>::lane(Fy, j);
      const unsigned long long s = (unsigned long long)__double_as_longlong(ux * ux + uy * uy);
      if (s > *(volatile unsigned long long *)out.max2) atomicMax(out.max2, s);
    }
}

// The fields as doubles; solid rows (written by the tile beside them) carry their
// ghost rho, psi, U and zeros.
template <class V, int R, class real>
__device__ __forceinline__ void emit(const Canon<real> &m, const Fields &out, const Window<V, R> &win,
                                     const real (&wrho)[R + 2][Val<V>::N * kH + 4], int w, int lane, int, int y,
                                     int x0, const bool (&act)[Val<V>::N], bool node, bool solid, real ss,
                                     const V (&f)[9], V r, bool) {
  constexpr int N = Val<V>::N;
  if (!node && !solid) return;
  V v[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) v[k] = Val<V>::bc((real)0);
  if (node) {
    V d13, d24, jx, jy;
    force(m, win, w, lane + 2, ss, v[2], v[3], v[4], v[5], v[6]);
    momentum(f, d13, d24, jx, jy);
    const V half = Val<V>::bc((real)0.5);
    v[0] = vfma(half, v[2], jx) / r;
    v[1] = vfma(half, v[3], jy) / r;
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (!act[j]) break;
    const size_t i = (size_t)y * m.nx + x0 + lane + j * kH;
    const bool ghost = solid && m.wetting != LBM_WET_MARTYS_CHEN;
    if (out.o[0]) out.o[0][i] = (double)(node || ghost ? wrho[w][lane + j * kH + 2] : (real)0);
    if (out.o[1]) out.o[1][i] = (double)Val<V>::lane(win.p[w][lane + 2], j);
    if (out.o[2]) out.o[2][i] = (double)Val<V>::lane(win.u[w][lane + 2], j);
#pragma unroll
    for (int k = 0; k < 7; ++k)
      if (out.o[3 + k]) out.o[3 + k][i] = (double)Val<V>::lane(v[k], j);
  }
}

// Tile of m.sw columns x R rows per CTA of R + 3 warps: warps 0 .. R + 1 each
// load one row (the tile's, the one above, the one below), the last one the
// columns beside the tile.  Window row w holds row y0 - 1 + w.
// CTAs per SM that the registers leave room for: 56 registers a thread in tiles of 8
// rows (with 62 and two CTAs FP64 at 400 x 200 took 103 us a step instead of 79) and
// of 4 (with 80 and three, FP32 at 2047 x 1025 59 instead of 45), 64 in those of 2.
constexpr int min_ctas(int R) { return R == 8 ? 3 : (R == 4 ? 5 : 6); }

template <class V, int R, class OUT>
__global__ void __launch_bounds__((R + 3) * 32, min_ctas(R))
    k_canon(Canon<typename Val<V>::R> m, const typename Val<V>::R *__restrict__ fin, OUT out,
            const double *__restrict__ coef, int *flag) {
  typedef typename Val<V>::R real;
  constexpr int N = Val<V>::N;
  static_assert(2 * (R + 2) + 4 <= 32, "one warp loads the columns beside the tile");
  __shared__ Window<V, R> win;
  __shared__ real wrho[R + 2][N * kH + 4];  // column c at c + 2
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int band = (int)(blockIdx.x / (unsigned)m.strips);
  const int x0 = ((int)blockIdx.x - band * m.strips) * m.sw, wr = min(m.sw, m.nx - x0);
  const int first = m.walls ? 1 : 0, last = m.walls ? m.ny - 1 : m.ny;  // fluid rows [first, last)
  const int y0 = first + band * R;
  const int nr = min(R, last - y0);
  const size_t n = (size_t)m.nx * m.ny;
  const bool geo = m.walls && m.wetting != LBM_WET_MARTYS_CHEN;
  const bool low = geo && y0 == 1, high = geo && y0 + nr == m.ny - 1;  // the tile touches a wall with a ghost row

  int w = warp, hc = 0;  // window row; column of a thread of the last warp
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
  const int v = y0 - 1 + w;
  const bool solid = m.walls && (v == 0 || v == m.ny - 1);
  const int y = v < 0 ? v + m.ny : (v >= m.ny ? v - m.ny : v);
  const bool row_warp = warp < R + 2;
  bool act[N];
#pragma unroll
  for (int j = 0; j < N; ++j) act[j] = lane + j * kH < wr;  // a later one implies the earlier
  int gx = x0 + hc;
  gx = gx < 0 ? gx + m.nx : (gx >= m.nx ? gx - m.nx : gx);

  // the wall coefficients of a ghost row, loaded before the densities it waits for
  double kc[N];
  if (on && solid && geo) {
    const double *c = coef + (m.n_iter > 0 ? 0 : 2 * m.nx) + (v != 0 ? m.nx : 0);
#pragma unroll
    for (int j = 0; j < N; ++j)
      if (row_warp ? act[j] : j == 0) kc[j] = c[row_warp ? x0 + lane + j * kH : gx];
  }
  bool bad = false, ok = true;
  V f[9], r = Val<V>::bc((real)0);
  if (on && (row_warp ? act[0] : true)) {
    if (!solid) {
      const real *q = fin + (size_t)y * m.nx + (row_warp ? x0 + lane : gx);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        f[a] = Val<V>::bc(q[a * n]);
        if (N == 2 && row_warp && act[N - 1]) Val<V>::set(f[a], 1, q[a * n + kH]);
      }
      r = f[0];
#pragma unroll
      for (int a = 1; a < 9; ++a) r = r + f[a];
      ok = plain(m, r);
      V psi, U;
      psi_U_plain(m, r, psi, U);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (row_warp ? act[j] : j == 0) {
          const int c = row_warp ? lane + j * kH : hc;
          const real rj = Val<V>::lane(r, j);
          bad |= !(rj > (real)0) || rj > m.rho_max;
          wrho[w][c + 2] = rj;
          win.put(w, c, Val<V>::lane(psi, j), Val<V>::lane(U, j));
        }
      }
    } else if (!geo) {  // Martys-Chen: psi = U = 0 on the solid rows
#pragma unroll
      for (int j = 0; j < N; ++j)
        if (row_warp ? act[j] : j == 0) win.put(w, row_warp ? lane + j * kH : hc, (real)0, (real)0);
    }
  }
  // densities out of the ordinary (none in a stable state) take the plain division
  // and root; decided for the CTA at the barrier, a branch for each thread in the
  // load phase cost 2 of 44 us at 2047 x 1025
  if constexpr (std::is_same<V, double>::value) {
    __syncthreads();
  } else if (__syncthreads_or(!ok)) {
    if (!ok) {
      V psi, U;
      psi_U(m, r, psi, U);
#pragma unroll
      for (int j = 0; j < N; ++j)
        if (row_warp ? act[j] : j == 0) win.put(w, row_warp ? lane + j * kH : hc, Val<V>::lane(psi, j), Val<V>::lane(U, j));
    }
    ok = false;
    __syncthreads();
  } else {
    ok = true;
  }
  if (low || high) {  // uniform in the CTA
    if (on && solid) {
      // v == 0 from window rows 1, 2; v == ny - 1 from the two rows below it
      const real *q1 = wrho[v != 0 ? w - 1 : 1], *q2 = wrho[v != 0 ? w - 2 : 2];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (row_warp ? act[j] : j == 0) {
          const int c = row_warp ? lane + j * kH : hc;
          real g, psi, U;
          ghost(m, q1[c + 1], q1[c + 2], q1[c + 3], q2[c + 2], (real)kc[j], g, psi, U);
          win.put(w, c, psi, U);
          if (std::is_same<OUT, Fields>::value) wrho[w][c + 2] = g;
        }
      }
    }
    __syncthreads();
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0 && *(volatile int *)flag == 0) atomicOr(flag, 1);
  const bool dn = m.walls && y == 1, up = m.walls && y == m.ny - 2;
  const real ss = dn ? m.ss_dn : (up ? m.ss_up : (real)0);
  const bool node = warp >= 1 && warp <= nr && act[0];
  emit(m, out, win, wrho, w, lane, warp, y, x0, act, node, solid && row_warp && on, ss, f, r, ok);
}

template <class V, int R, class OUT>
cudaError_t launch(const lbm_ctx *C, const void *src, OUT out) {
  typedef typename Val<V>::R real;
  Canon<real> m(C);
  const int W = Val<V>::N * kH;
  m.strips = (C->nx + W - 1) / W;
  m.sw = Val<V>::N == 1 ? (C->nx + m.strips - 1) / m.strips : W;
  const int nrows = C->walls ? C->ny - 2 : C->ny;
  const unsigned grid = (unsigned)m.strips * (unsigned)((nrows + R - 1) / R);
  k_canon<V, R, OUT><<<grid, (R + 3) * 32, 0, C->stream>>>(m, (const real *)src, out, C->d_coef, C->d_flag);
  return cudaGetLastError();
}

}  // namespace

// Rows per tile.  FP32: 4 (2047 x 1025: 56 us per step, with 2 rows 63, with 6
// rows 62).  FP64: the FP64 pipe of an SM quarter takes 64 cycles for an
// operation of a warp, so small domains take as long as one warp's chain (100 x
// 60: 16.7 us) and want few rows per CTA; larger ones are bound by the pipe and
// want few repeated rows: 2 / 8 rows, 200 x 100 27.7 / 30.3, 400 x 200 79.8 /
// 79.1, 800 x 400 253 / 230 us.
cudaError_t lbm_canon_step(const lbm_ctx *C, const void *src, void *dst, unsigned long long *launches) {
  ++*launches;
  if (C->precision == 32) return launch<F2, 4>(C, src, Step<float>{(float *)dst});
  const Step<double> out{(double *)dst};
  return (long long)C->nx * C->ny < 80000 ? launch<double, 2>(C, src, out) : launch<double, 8>(C, src, out);
}

// The getters' fields and the largest speed, in one pass over the populations
// (before: fields, then seven planes of doubles, then the reduction of two of
// them).  4096 x 2048: largest speed, a call, 609 -> 169 us.
cudaError_t lbm_canon_fields(const lbm_ctx *C, const void *f, double *const (&o)[10], unsigned long long *launches) {
  ++*launches;
  Fields out;
  for (int k = 0; k < 10; ++k) out.o[k] = o[k];
  return C->precision == 32 ? launch<F2, 4>(C, f, out) : launch<double, 4>(C, f, out);
}

cudaError_t lbm_canon_max_speed2(const lbm_ctx *C, const void *f, double *max2, unsigned long long *launches) {
  ++*launches;
  const cudaError_t e = cudaMemsetAsync(max2, 0, sizeof(double), C->stream);
  if (e != cudaSuccess) return e;
  const Speed out{(unsigned long long *)max2};
  return C->precision == 32 ? launch<F2, 4>(C, f, out) : launch<double, 4>(C, f, out);
}
